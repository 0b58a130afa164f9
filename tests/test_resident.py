"""The on-chip 2D stepper (default plan of 2D complex-float contexts) against
the FP64 oracle and against the sweep launches: smallest tiles, remainders,
every halo width, both modes, schedules, shares of the norm out of their
first range.

Tolerances.  A step rounds every point a few times (2^-24 relative each, of
which the H1 factor, the two changes and the pending scale are added to psi
once): 4 x 6e-8 per step, added up linearly over the steps as a bound.
"""
import numpy as np
import pytest

import oracle
from paper_1906_06327_gb300 import inputs
from paper_1906_06327_gb300.rotgp import Solver

pytestmark = pytest.mark.gpu

STEPS = 12
TOL = 4 * 6e-8 * STEPS
KW = dict(gamma=1.0, nu=1.1, g=60.0, omega=0.6)


def _rel(a, b):
    return np.linalg.norm(a - b) / np.linalg.norm(b)


def _smooth(n, h, seed):
    """A state of a few oracle steps from the seeded start (the first steps of
    a random-phase state lose most of its norm)."""
    grid, phys = oracle.Grid(n, h), oracle.Phys(dt=2e-3, **KW)
    psi = oracle.init_analytic(grid, 1, inputs.random_phase_field(n[0], n[1], seed))
    return oracle.steps(grid, phys, psi, 30, True)[0].astype(np.complex64)


# (grid, kappa = dt / (4 h^2)): halos of 4, 6 and 14 points; one tile, two
# tiles, a last tile of one odd column, many tiles, more points than threads
CASES = [((10, 10), 0.006), ((14, 15), 0.02), ((30, 31), 0.1), ((16, 29), 0.02),
         ((37, 50), 0.02), ((129, 64), 0.006), ((201, 135), 0.02), ((160, 96), 0.12),
         ((333, 290), 0.02), ((640, 420), 0.02)]


@pytest.mark.parametrize("imag", [True, False])
@pytest.mark.parametrize("n,kappa", CASES)
def test_steps_match_oracle(n, kappa, imag):
    h = (12.0 / n[0], 11.0 / n[1])
    dt = 4.0 * kappa * min(h) ** 2
    psi = _smooth(n, h, 3)
    ref, _ = oracle.steps(oracle.Grid(n, h), oracle.Phys(dt=dt, **KW), psi.astype(np.complex128),
                          STEPS, imag)
    s = Solver(n, h, dt=dt, **KW)
    s.set_psi(psi)
    s.step_imag(5) if imag else s.step_real(5)
    s.step_imag(STEPS - 5) if imag else s.step_real(STEPS - 5)
    got = s.get_psi()
    assert _rel(got, ref) < TOL, _rel(got, ref)
    assert s.observables()["step"] == STEPS
    for edge in (got[0], got[-1], got[:, 0], got[:, -1]):
        assert not edge.any()


@pytest.mark.parametrize("imag", [True, False])
def test_schedule_matches_sweep_launches(imag):
    n, h = (70, 53), (0.2, 0.22)
    om = np.linspace(0.6, 0.5, 70)  # more than one table build
    psi = _smooth(n, h, 4)
    a, b = Solver(n, h, dt=1e-3, **KW), Solver(n, h, dt=1e-3, **KW)
    for ax in (0, 1):
        b.set_solver(ax, "thomas")  # a form asked for: the sweep launches
    for s in (a, b):
        s.set_psi(psi)
        s.step_schedule(om, imag=imag)
        s.step_real(1)
    assert _rel(a.get_psi(), b.get_psi()) < 2 * 4 * 6e-8 * (len(om) + 1)


@pytest.mark.parametrize("scale", [1e-6, 3e5])
def test_norm_far_from_one(scale):
    """The shares of the norm start out scaled for unit norm."""
    n, h = (60, 44), (0.2, 0.25)
    psi = _smooth(n, h, 5)
    kw = dict(KW, g=0.0)
    a, b = Solver(n, h, dt=1e-3, **kw), Solver(n, h, dt=1e-3, **kw)
    a.set_psi(psi)
    b.set_psi((psi * np.float32(scale)).astype(np.complex64))
    for s in (a, b):
        s.step_real(3)
    na, nb = a.observables()["norm"], b.observables()["norm"]
    assert abs(nb / (na * float(np.float32(scale)) ** 2) - 1) < 1e-6
    for s in (a, b):
        s.step_imag(3)
    assert abs(b.observables()["norm"] - 1) < 1e-6
    assert _rel(b.get_psi(), a.get_psi()) < TOL


def test_nan_state_is_reported():
    from paper_1906_06327_gb300.rotgp import RotgpError
    n, h = (60, 44), (0.2, 0.25)
    psi = _smooth(n, h, 6)
    psi[20, 20] = np.nan
    s = Solver(n, h, dt=1e-3, **KW)
    s.set_psi(psi)
    s.step_imag(2)
    with pytest.raises(RotgpError):
        s.sync()
