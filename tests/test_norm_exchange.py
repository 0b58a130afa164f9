"""The grid-wide exchange of the norm in the cooperative 2D steppers: totals far
from the one before them (random-phase starts lose most of their norm in the
first step and little in the second), and totals that no scale of the shares
holds at once.

The on-chip stepper's tiles fill their CTAs from about 560 to 1,100 points a
side: every thread then has a share, and the sums of a CTA are at their largest.

Tolerances: complex double as tests/test_double_steps.py, 2e-15 per step against
the chunked sweeps; complex float as tests/test_resident.py, 4 x 6e-8 per step
and form, and the norm of a renormalised state within 1e-6."""
import numpy as np
import pytest

import oracle
from paper_1906_06327_gb300 import inputs
from paper_1906_06327_gb300.rotgp import RotgpError, Solver

KW = dict(gamma=1.0, nu=1.1, lam=1.3, g=60.0, omega=0.5)


def _start(n, seed):
    return oracle.init_analytic(oracle.Grid(n, (12.0 / n[0], 12.0 / n[1])), 1,
                                inputs.random_phase_field(n[0], n[1], seed))


@pytest.mark.gpu
@pytest.mark.parametrize("n,kappa", [((300, 300), 0.5), ((128, 128), 0.45), ((64, 64), 0.3),
                                     ((40, 33), 0.35)])
def test_double_steps_through_a_jump_of_the_norm(n, kappa):
    """The second total is several times the first, beyond the scale that the
    first one left."""
    h = tuple(12.0 / v for v in n)
    dt = 4.0 * kappa * min(h) ** 2
    psi = _start(n, 3)
    s, t = (Solver(n, h, dt=dt, precision="fp64", **KW) for _ in range(2))
    for ax in (0, 1):
        t.set_solver(ax, "thomas")
    for x in (s, t):
        x.set_psi(psi, normalise=True)
        x.step_imag(6)
    ref = t.get_psi()
    assert np.linalg.norm(s.get_psi() - ref) < 2e-15 * 6 * np.linalg.norm(ref)
    assert abs(s.observables()["norm"] - 1) < 1e-14


@pytest.mark.gpu
@pytest.mark.parametrize("precision,scale", [("fp64", 1e-120), ("fp64", 1e100), ("fp64", 3e-8),
                                             ("fp32", 1e-12), ("fp32", 1e9)])
def test_first_total_far_out_of_range(precision, scale):
    n, h = (90, 70), (0.13, 0.17)
    kw = dict(KW, g=0.0)
    psi = _start(n, 4)
    if precision == "fp32":
        psi = psi.astype(np.complex64)
    res = []
    for f in (1.0, scale):
        s = Solver(n, h, dt=1e-3, precision=precision, **kw)
        s.set_psi((psi * f).astype(psi.dtype))
        s.step_imag(5)
        res.append(s.get_psi())
    tol = 1e-13 if precision == "fp64" else 5 * 4 * 6e-8
    assert np.linalg.norm(res[1] - res[0]) < tol * np.linalg.norm(res[0])


@pytest.mark.gpu
@pytest.mark.parametrize("precision", ["fp64", "fp32"])
def test_zero_state_ends_in_an_error(precision):
    n = (60, 45)
    s = Solver(n, (0.2, 0.25), dt=1e-3, precision=precision, **KW)
    s.set_psi(np.zeros((46, 61), np.complex128 if precision == "fp64" else np.complex64))
    s.step_imag(3)
    with pytest.raises(RotgpError):
        s.sync()


# one to three segments a thread, both short halos; 384 threads (halo above 8)
FULL = [((560, 560), 0.006), ((600, 600), 0.006), ((600, 600), 0.02), ((800, 800), 0.006),
        ((800, 800), 0.02), ((900, 900), 0.02), ((1024, 1024), 0.006), ((1100, 1100), 0.02),
        ((1024, 768), 0.02), ((1000, 1000), 0.1)]


def _flat(n):
    """Density everywhere on the grid, a phase that varies slowly."""
    x, y = np.meshgrid(np.linspace(0, 1, n[0] + 1), np.linspace(0, 1, n[1] + 1))
    psi = np.exp(2j * np.pi * (x - 2 * y)) * (1 + 0.2 * np.sin(7 * x) * np.cos(5 * y))
    psi[[0, -1]] = 0
    psi[:, [0, -1]] = 0
    return (psi / 12.0).astype(np.complex64)  # norm 1 on 12 x 12, to a few percent


def _pair(n, kappa):
    h = (12.0 / n[0], 12.0 / n[1])
    s, t = (Solver(n, h, dt=4.0 * kappa * min(h) ** 2, **KW) for _ in range(2))
    for ax in (0, 1):
        t.set_solver(ax, "thomas")  # the sweep launches
    return s, t


@pytest.mark.gpu
@pytest.mark.parametrize("n,kappa", FULL)
def test_full_tiles_norm(n, kappa):
    s, t = _pair(n, kappa)
    for x in (s, t):
        x.set_psi(_flat(n), normalise=True)
        x.step_imag(1)
    assert abs(s.observables()["norm"] - 1) < 1e-6
    for x in (s, t):
        x.step_imag(19)
        x.step_real(5)
    assert abs(s.observables()["norm"] - 1) < 1e-6
    ref = t.get_psi()
    assert np.linalg.norm(s.get_psi() - ref) < 2 * 4 * 6e-8 * 25 * np.linalg.norm(ref)


@pytest.mark.gpu
@pytest.mark.parametrize("n", [(800, 800), (1000, 1000)])
def test_full_tiles_report_a_nan(n):
    s, _ = _pair(n, 0.02)
    psi = _flat(n)
    psi[n[1] // 2, n[0] // 3] = np.nan
    s.set_psi(psi)
    s.step_imag(200)
    with pytest.raises(RotgpError):
        s.sync()


@pytest.mark.gpu
@pytest.mark.parametrize("scale", [1e3, 1e6])
def test_full_tiles_normalise_a_large_state(scale):
    """Shares of every thread beyond the first scale (a norm of 1e6 and 1e12)."""
    n = (800, 800)
    s, t = _pair(n, 0.02)
    psi = _flat(n)
    for x, f in ((s, scale), (t, 1.0)):
        x.set_phys(g=0.0)
        x.set_psi((psi * np.float32(f)).astype(np.complex64))
        x.step_imag(4)
    assert abs(s.observables()["norm"] - 1) < 1e-6
    ref = t.get_psi()
    assert np.linalg.norm(s.get_psi() - ref) < 2 * 4 * 6e-8 * 4 * np.linalg.norm(ref)


@pytest.mark.gpu
@pytest.mark.parametrize("norm", [0.9, 1.9, 2.7, 3.8, 7.5])
def test_first_norm_in_one_point(norm):
    """A share as large as a total may be: the state in one point, the scale of
    the shares just above 1 / (h_x h_y), Delta too short to spread it (odd N_x: a
    single step that runs in the stepper)."""
    n, h = (61, 44), (0.25, 0.2505)
    psi = np.zeros((n[1] + 1, n[0] + 1), np.complex64)
    psi[20, 30] = np.sqrt(norm / (h[0] * h[1]))
    s = Solver(n, h, gamma=1.0, nu=1.0, g=0.0, omega=0.0, dt=1e-9)
    s.set_psi(psi)
    s.step_imag(1)
    assert abs(s.observables()["norm"] - 1) < 1e-6
