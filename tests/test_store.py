"""Reading a state back into complex float: values that are not finite come back as
they were loaded."""
import numpy as np
import pytest

from paper_1906_06327_gb300.rotgp import Solver

pytestmark = pytest.mark.gpu


def test_infinities_come_back_as_loaded():
    n = (40, 30)
    psi = np.zeros((31, 41), np.complex64)
    psi[10, 10] = 1.0
    psi[11, 12] = complex(np.inf, 2.0)
    psi[13, 14] = complex(-np.inf, np.nan)
    s = Solver(n, (0.3, 0.3), dt=1e-3, g=1.0)
    s.set_psi(psi)
    got = s.get_psi(fp64=False)
    assert np.array_equal(got.view(np.float32), psi.view(np.float32), equal_nan=True)



@pytest.mark.parametrize("n", [(4, 5), (15, 16), (16, 15), (255, 9), (256, 9), (257, 8), (5, 4, 70),
                               (20, 31, 33), (33, 40, 6)])
@pytest.mark.parametrize("precision", ["fp32", "fp64"])
def test_copies_between_all_types(n, precision):
    """Loading and reading back, with and without renormalisation, around the
    lengths at which rows are split and copied point by point."""
    rng = np.random.default_rng(3)
    shape = tuple(v + 1 for v in reversed(n))
    inner = np.zeros(shape)
    inner[tuple(slice(1, -1) for _ in n)] = 1
    work = np.complex64 if precision == "fp32" else np.complex128
    h = (0.3, 0.25, 0.2)[:len(n)]
    s = Solver(n, h, dt=1e-3, precision=precision)
    for dt in (np.complex64, np.complex128):
        psi = (rng.normal(size=shape) + 1j * rng.normal(size=shape)).astype(dt)
        s.set_psi(psi)
        want = (psi * inner).astype(work)
        assert np.array_equal(s.get_psi(fp64=True), want.astype(np.complex128))
        assert np.array_equal(s.get_psi(fp64=False), want.astype(np.complex64))
        s.set_psi(psi, normalise=True)
        ref = want.astype(np.complex128)
        ref /= np.sqrt(np.prod(h) * (np.abs(ref) ** 2).sum())
        eps = 2.0**-23 if precision == "fp32" else 1e-15
        assert np.abs(s.get_psi(fp64=True) - ref).max() < eps * np.abs(ref).max()
        assert np.abs(s.get_psi(fp64=False) - ref).max() < 2.0**-23 * np.abs(ref).max()


@pytest.mark.parametrize("precision", ["fp32", "fp64"])
def test_short_rows_cost_no_more_than_long_ones(precision):
    """As many points of complex double in rows of 20 as in rows of 300."""
    torch = pytest.importorskip("torch")
    us = {}
    for n in ((20, 300, 300), (300, 300, 20)):
        s = Solver(n, (0.1,) * 3, dt=1e-3, precision=precision)
        s.init_analytic(1, seed=1)
        out = torch.zeros(s.shape, dtype=torch.complex128, device="cuda")
        s.get_psi(out)
        s.profile(True)
        s.profile_read()
        for _ in range(10):
            s.get_psi(out)
            s.set_psi(out, normalise=True)
        us[n] = sum(r["total_ms"] for r in s.profile_read().values())
        s.close()
    assert us[(20, 300, 300)] < 2.0 * us[(300, 300, 20)], us
