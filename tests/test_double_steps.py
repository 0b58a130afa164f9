"""Imaginary time in complex double (the default plan): blocks of 2D steps in
one launch, and the row and column sweeps of larger and 3D states, at sizes
around the edges of their splits (points per lane, lines per CTA, segments and
halos of the columns), for short and long halos, against the chunked sweeps
that an explicitly chosen form still takes, and loosely against the oracle.

Tolerance: a step rounds a point some ten times at 1.1e-16 relative, and the
scale once: 2e-15 per step, added up linearly.  (Both forms are up to 2e-14
per step from the oracle, by the same amount: coordinates and potential are
rounded differently there.)"""
import numpy as np
import pytest

import oracle
from paper_1906_06327_gb300 import inputs
from paper_1906_06327_gb300.rotgp import Solver

pytestmark = pytest.mark.gpu

STEPS = 6
KW = dict(gamma=1.0, nu=1.1, lam=1.3, g=60.0, omega=0.6)


# (grid, kappa of the first axis): 1 to 8 points per lane on either axis, one
# and several lines per CTA; halos of 9, 12, 20 and 50 points; segments that
# do not divide a line, a line shorter than its halo, partial groups of columns
CASES = [((4, 5), 0.02), ((31, 33), 0.02), ((128, 129), 0.006), ((200, 130), 0.02),
         ((140, 520), 0.02), ((700, 60), 0.08), ((300, 257), 0.02), ((64, 96), 0.25),
         ((1100, 40), 0.02), ((5, 7, 6), 0.02), ((33, 20, 40), 0.02), ((130, 31, 97), 0.02),
         ((40, 257, 14), 0.0005), ((20, 150, 120), 0.004), ((260, 12, 33), 0.006)]


@pytest.mark.parametrize("n,kappa", CASES)
def test_steps_match_chunked_sweeps(n, kappa):
    h = tuple(10.0 / v for v in n)
    dt = 4.0 * kappa * h[0] ** 2
    grid, phys = oracle.Grid(n, h), oracle.Phys(dt=dt, **KW)
    psi = oracle.init_analytic(grid, 1, inputs.random_phase_field(n[0], n[1], 2))
    s = Solver(n, h, dt=dt, precision="fp64", **KW)
    s.set_psi(psi, normalise=True)
    s.step_imag(2)
    s.step_imag(STEPS - 2)
    got = s.get_psi()
    t = Solver(n, h, dt=dt, precision="fp64", **KW)
    for ax in range(len(n)):
        t.set_solver(ax, "thomas")
    t.set_psi(psi, normalise=True)
    t.step_imag(STEPS)
    ref = t.get_psi()
    err = np.linalg.norm(got - ref) / np.linalg.norm(ref)
    assert err < 2e-15 * STEPS, err
    ref, _ = oracle.steps(grid, phys, psi / np.sqrt(oracle.norm(grid, psi)), STEPS, True)
    assert np.linalg.norm(got - ref) < 1e-10 * np.linalg.norm(ref)
    assert abs(s.observables()["norm"] - 1) < 1e-14


def test_scale_of_the_state_does_not_matter():
    """The shares of the norm start out scaled for unit norm."""
    n, h = (60, 45), (0.2, 0.25)
    grid = oracle.Grid(n, h)
    psi = oracle.init_analytic(grid, 1, inputs.random_phase_field(n[0], n[1], 3))
    kw = dict(KW, g=0.0)
    ref = None
    for f in (1.0, 1e-40, 3e60):
        s = Solver(n, h, dt=1e-3, precision="fp64", **kw)
        s.set_psi(psi * f)
        s.step_imag(5)
        got = s.get_psi()
        ref = got if ref is None else ref
        assert np.linalg.norm(got - ref) < 1e-14 * np.linalg.norm(ref)
