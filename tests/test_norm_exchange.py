"""The grid-wide exchange of the norm in the cooperative 2D steppers: totals far
from the one before them (random-phase starts lose most of their norm in the
first step and little in the second), and totals that no scale of the shares
holds at once.

Tolerances: complex double as tests/test_double_steps.py, 2e-15 per step against
the chunked sweeps."""
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
