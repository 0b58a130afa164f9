"""Real time in the one-line-per-lane TMA sweeps of complex float (the default
of even rows in 3D up to kappa = 0.005) and beyond it against the FP64 oracle: groups of lines and chunks partly
outside the grid, one and several segments per line, both chunk lengths, every
ring depth.

Tolerance as for the other sweeps of complex float: a point is rounded twice
per sweep and step at 6e-8, added up linearly."""
import numpy as np
import pytest

import oracle
from paper_1906_06327_gb300 import inputs
from paper_1906_06327_gb300.rotgp import Solver

pytestmark = pytest.mark.gpu

STEPS = 10
KW = dict(gamma=1.0, nu=1.1, lam=1.3, g=60.0, omega=0.6)

# (grid, (chunk, ring, segments) or the default plan)
CASES = [((32, 32, 32), None), ((34, 33, 31), None), ((130, 17, 70), None), ((18, 259, 20), None),
         ((96, 40, 41), (8, 3, 1)), ((96, 40, 41), (8, 4, 3)), ((66, 40, 50), (8, 6, 2)),
         ((66, 40, 50), (16, 3, 2)), ((70, 34, 49), (16, 4, 1)), ((302, 130), (8, 5, 3))]


@pytest.mark.parametrize("kappa", [0.0045, 0.02])
@pytest.mark.parametrize("n,shape", CASES)
def test_real_time_matches_oracle(n, shape, kappa):
    h = tuple(10.0 / max(n) * f for f in (1.0, 1.02, 1.05))[:len(n)]
    dt = 4.0 * kappa * h[0] ** 2
    grid = oracle.Grid(n, h)
    psi = oracle.init_analytic(grid, 1, inputs.random_phase_field(n[0], n[1], 3))
    psi = oracle.steps(grid, oracle.Phys(dt=min(dt, 2e-3), **KW), psi, 20, True)[0]
    psi = psi.astype(np.complex64)
    ref, _ = oracle.steps(grid, oracle.Phys(dt=dt, **KW), psi.astype(np.complex128), STEPS, False)
    s = Solver(n, h, dt=dt, **KW)
    for ax in range(len(n) if shape else 0):
        s.tune(ax, 1, shape[0], shape[1], 1, shape[2])
    s.set_psi(psi)
    s.step_real(STEPS)
    got = s.get_psi()
    err = np.linalg.norm(got - ref) / np.linalg.norm(ref)
    assert err < 2 * len(n) * 6e-8 * STEPS, err
    for ax in range(len(n)):
        assert not np.take(got, (0, -1), axis=ax).any()
