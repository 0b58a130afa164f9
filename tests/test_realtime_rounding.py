"""Norm and state of complex-float real time on smooth states whose changes per step
are a few units of the last place (fine grids, short steps), in each form that adds a
point to its change once: the on-chip stepper, tiles on odd rows, the centred TMA
sweeps.

Bounds: 400 steps, a few unbiased roundings of 2^-24 relative per point and step,
independent of each other: the norm of 1e4 points and more moves by far less than
4e-10 per step, and psi by at most 4 x 2^-24 x sqrt(roundings), taken as 5e-6 (a
rounding that is the same at a point every step gives 1e-5 and more, and 2e-9 to 8e-9
per step)."""
import numpy as np
import pytest

from paper_1906_06327_gb300.rotgp import Solver

pytestmark = pytest.mark.gpu

STEPS = 400


@pytest.mark.parametrize("kappa", [0.0005, 0.0025, 0.0045])
@pytest.mark.parametrize("n,form", [((256, 256), None), ((255, 255, 24), None),
                                    ((256, 256, 24), None), ((1400, 1100), "thomas")])
def test_small_changes_are_rounded_without_bias(n, form, kappa):
    h = tuple(12.0 / v for v in n)
    kw = dict(gamma=1.0, nu=1.05, lam=1.2, g=0.0, omega=0.3, dt=4 * kappa * h[0] ** 2)
    s = Solver(n, h, **kw)
    for ax in range(len(n) if form else 0):
        s.set_solver(ax, form)
    s.init_analytic(1)
    psi = s.get_psi(fp64=False)
    s.set_psi(psi, normalise=True)
    s.step_real(1)
    n0, psi = s.observables()["norm"], s.get_psi(fp64=False)
    s.step_real(STEPS)
    assert abs(s.observables()["norm"] - n0) < 4e-10 * STEPS
    t = Solver(n, h, precision="fp64", **kw)
    t.set_psi(psi)
    t.step_real(STEPS)
    ref = t.get_psi()
    assert np.linalg.norm(s.get_psi() - ref) < 5e-6 * np.linalg.norm(ref)


@pytest.mark.parametrize("n,kappa,per_step", [((128, 128), 0.0005, 4e-10),
                                              ((128, 128), 0.01, 1.3e-9),
                                              ((256, 256), 0.01, 1.3e-9)])
@pytest.mark.parametrize("omega", [0.0, 0.7])
def test_exact_solve_joins_its_carries_without_bias(n, kappa, per_step, omega):
    """Carries below half a unit of the last place are not lost.  Bounds: as above, or
    eight times the rms effect of rounded weights (8e-7 kappa^2 an axis)."""
    h = (12.0 / n[0],) * 2
    s = Solver(n, h, gamma=1.0, nu=1.05, g=0.0, omega=omega, dt=4 * kappa * h[0] ** 2)
    for ax in (0, 1):
        s.set_solver(ax, "hybrid")
    s.init_analytic(1)
    s.step_imag(2)
    s.step_real(1)
    n0 = s.observables()["norm"]
    s.step_real(STEPS)
    assert abs(s.observables()["norm"] - n0) < per_step * STEPS
