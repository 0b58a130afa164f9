"""Forms and shapes that were asked for are the ones that run: contexts whose
default plan takes kernels of its own (tiles with long halos, the on-chip stepper)
against contexts with the same forms asked for from the start, bit for bit."""
import numpy as np
import pytest

from paper_1906_06327_gb300.rotgp import Solver

pytestmark = pytest.mark.gpu

KW = dict(gamma=1.0, nu=1.1, g=20.0, omega=0.4)


def _run(s, imag=True):
    s.init_analytic(1, seed=4)
    s.step_imag(3) if imag else s.step_real(3)
    return s.get_psi()


@pytest.mark.parametrize("imag", [True, False])
def test_tuned_exact_solve_runs(imag):
    """A halo of 32 points: the exact solve is the form that rotgp_tune shapes,
    the default runs tiles."""
    n, h = (300, 300), (0.1, 0.1)
    a, b = (Solver(n, h, dt=4 * 1.15 * 0.01, **KW) for _ in range(2))
    for ax in (0, 1):
        b.set_solver(ax, "hybrid")
    for s in (a, b):
        for ax in (0, 1):
            s.tune(ax, 1, 8, 3, 1, 2)
        assert s.info()["hybrid_cluster"] == [2, 2]
    assert np.array_equal(_run(a, imag), _run(b, imag))


@pytest.mark.parametrize("n,kappa", [((256, 20, 256), 1.15), ((128, 96), 0.1)])
def test_autotune_that_keeps_the_default_plan(n, kappa):
    """The default plan as it was timed: 3D tiles on x and z with the exact solve on
    a y axis shorter than the halo (34 points); the on-chip stepper.  (They are
    the faster ones by 10% and several times.)"""
    h = (0.1,) * len(n)
    kw = dict(KW, lam=1.0, dt=4 * kappa * 0.01)
    a, b = Solver(n, h, **kw), Solver(n, h, **kw)
    a.init_analytic(1, seed=4)
    if a.autotune(20)["choice"] != 0:
        pytest.skip("a sweep form was the faster one")
    assert a.info() == b.info()
    assert np.array_equal(_run(a), _run(b))
    assert np.array_equal(_run(a, False), _run(b, False))


@pytest.mark.parametrize("n,kappa", [((32, 32), 0.5), ((64, 64), 1.15), ((63, 65), 1.15),
                                     ((48, 48, 48), 1.15)])
def test_short_lines_with_long_halos_take_the_exact_solve(n, kappa):
    """Where tiles of tails would be the slower ones."""
    kw = dict(KW, lam=1.0, dt=4 * kappa * 0.01)
    a, b = (Solver(n, (0.1,) * len(n), **kw) for _ in range(2))
    for ax in range(len(n)):
        b.set_solver(ax, "hybrid")
    assert np.array_equal(_run(a), _run(b))
    assert np.array_equal(_run(a, False), _run(b, False))


def test_calls_of_one_step_take_the_sweeps():
    a, b = (Solver((64, 48), (0.2, 0.2), dt=1e-3, **KW) for _ in range(2))
    for ax in (0, 1):
        b.set_solver(ax, "thomas")
    for s in (a, b):
        s.init_analytic(1, seed=4)
        for _ in range(5):
            s.step_imag(1)
    assert np.array_equal(a.get_psi(), b.get_psi())


def test_complex_double_weights_follow_the_physics():
    """Built by the first imaginary-time step after a change: changes of Omega and
    Delta between steps, in schedules, in real time and in captured graphs."""
    from paper_1906_06327_gb300.rotgp import Batch
    n, h = (48, 40), (0.25, 0.28)
    a = Solver(n, h, dt=1e-3, precision="fp64", **KW)
    b = Batch([dict(n=n, h=h, dt=1e-3, **KW)] * 2, precision="fp64")
    for s in (a, *b.instances):
        s.init_analytic(1, seed=4)
        s.step_imag(2)
        s.set_phys(omega=0.3, dt=8e-4)
    a.step_imag(3)
    b.step_imag(3, mode="graph")
    for s in (a, *b.instances):
        s.step_schedule(np.array([0.3, 0.25, 0.2]), imag=True)
        s.step_schedule(np.array([0.2, 0.3]), imag=False)
        s.set_omega(0.1)
    a.step_imag(3)
    b.step_imag(3, mode="graph")
    a.set_omega(0.4)
    for s in b.instances:
        s.set_omega(0.4)
    a.step_imag(6)
    b.step_imag(3, mode="graph")
    b.step_imag(3, mode="graph")
    t = Solver(n, h, dt=1e-3, precision="fp64", **KW)
    for ax in (0, 1):
        t.set_solver(ax, "thomas")
    t.init_analytic(1, seed=4)
    t.step_imag(2)
    t.set_phys(omega=0.3, dt=8e-4)
    t.step_imag(3)
    t.step_schedule(np.array([0.3, 0.25, 0.2]), imag=True)
    t.step_schedule(np.array([0.2, 0.3]), imag=False)
    t.set_omega(0.1)
    t.step_imag(3)
    t.set_omega(0.4)
    t.step_imag(6)
    b.sync()
    ref = t.get_psi()
    for s in (a, *b.instances):
        assert np.linalg.norm(s.get_psi() - ref) < 2e-15 * 20 * np.linalg.norm(ref)
    # real time does not build them: one table launch per axis and mode
    a.profile(True)
    a.profile_read()
    a.set_omega(0.2)
    a.step_real(1)
    assert a.profile_read()["tables"]["launches"] == 4
    b.close()


@pytest.mark.parametrize("precision", ["fp32", "fp64"])
def test_observables_are_timed_by_kernel(precision):
    s = Solver((64, 48), (0.2, 0.2), dt=1e-3, precision=precision, **KW)
    s.init_analytic(1, seed=4)
    s.profile(True)
    s.profile_read()
    s.observables()
    rec = s.profile_read()
    assert rec["observables"]["launches"] == 1 and rec["vortex_count"]["launches"] == 1
