"""The tiled two-tail sweeps of complex float (the default plan where the halo
is above 16 points, in 3D real time and on odd rows) against the FP64 oracle:
one and several tiles per line, tiles and groups of lines partly outside the
grid, halos from a few points to 60, lines barely longer than the halo.

Tolerance as for the on-chip stepper, per sweep: every point is rounded a few
times per step at 6e-8, added up linearly; one more sweep in 3D."""
import numpy as np
import pytest

import oracle
from paper_1906_06327_gb300 import inputs
from paper_1906_06327_gb300.rotgp import Solver

pytestmark = pytest.mark.gpu

STEPS = 10
KW = dict(gamma=1.0, nu=1.1, lam=1.3, g=60.0, omega=0.6)

# (grid, kappa of the finest axis, imaginary time)
CASES = [((64, 70), 0.3, True), ((64, 70), 0.3, False), ((300, 77), 0.4, True),
         ((262, 515), 0.25, True), ((262, 515), 0.25, False), ((129, 128), 2.5, True),
         ((33, 20, 40), 0.02, True), ((33, 20, 40), 0.02, False), ((70, 64, 131), 0.02, False),
         ((40, 300, 33), 0.02, False), ((301, 17, 50), 0.02, True), ((96, 65, 34), 0.2, False),
         ((12, 33, 257), 0.006, False)]


@pytest.mark.parametrize("n,kappa,imag", CASES)
def test_steps_match_oracle(n, kappa, imag):
    h = tuple(10.0 / max(n) * f for f in (1.0, 1.02, 1.05))[:len(n)]
    dt = 4.0 * kappa * h[0] ** 2
    grid = oracle.Grid(n, h)
    psi = oracle.init_analytic(grid, 1, inputs.random_phase_field(n[0], n[1], 3))
    psi = oracle.steps(grid, oracle.Phys(dt=min(dt, 2e-3), **KW), psi, 20, True)[0]
    psi = psi.astype(np.complex64)
    ref, _ = oracle.steps(grid, oracle.Phys(dt=dt, **KW), psi.astype(np.complex128), STEPS, imag)
    s = Solver(n, h, dt=dt, **KW)
    s.set_psi(psi)
    s.step_imag(STEPS) if imag else s.step_real(STEPS)
    got = s.get_psi()
    err = np.linalg.norm(got - ref) / np.linalg.norm(ref)
    assert err < 2 * len(n) * 6e-8 * STEPS, err
    for ax in range(len(n)):
        assert not np.take(got, (0, -1), axis=ax).any()
    if imag:
        assert abs(s.observables()["norm"] - 1) < 1e-6
