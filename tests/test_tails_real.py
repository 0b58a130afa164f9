"""Real time in two-tail tiles on odd rows with short halos (3D), one and several tiles
per line on each axis, against the FP64 oracle, and the norm of such a run.

Tolerance as tests/test_tails.py: 6e-8 per rounding, two per sweep and step."""
import numpy as np
import pytest

import oracle
from paper_1906_06327_gb300 import inputs
from paper_1906_06327_gb300.rotgp import Solver

pytestmark = pytest.mark.gpu

STEPS = 10
KW = dict(gamma=1.0, nu=1.1, lam=1.3, g=60.0, omega=0.6)


@pytest.mark.parametrize("n,kappa", [((71, 64, 131), 0.02), ((41, 300, 33), 0.02),
                                     ((13, 33, 257), 0.006), ((301, 20, 18), 0.1)])
def test_odd_rows_match_oracle(n, kappa):
    h = tuple(10.0 / max(n) * f for f in (1.0, 1.02, 1.05))
    dt = 4.0 * kappa * h[0] ** 2
    grid = oracle.Grid(n, h)
    psi = oracle.init_analytic(grid, 1, inputs.random_phase_field(n[0], n[1], 3))
    psi = oracle.steps(grid, oracle.Phys(dt=min(dt, 2e-3), **KW), psi, 20, True)[0]
    psi = psi.astype(np.complex64)
    ref, norm = oracle.steps(grid, oracle.Phys(dt=dt, **KW), psi.astype(np.complex128), STEPS, False)
    s = Solver(n, h, dt=dt, **KW)
    s.set_psi(psi)
    s.step_real(STEPS)
    got = s.get_psi()
    assert np.linalg.norm(got - ref) < 2 * 3 * 6e-8 * STEPS * np.linalg.norm(ref)
    for ax in range(3):
        assert not np.take(got, (0, -1), axis=ax).any()
    assert abs(s.observables()["norm"] - oracle.norm(grid, ref)) < 1e-6
