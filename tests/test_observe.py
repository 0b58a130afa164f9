"""Observables, vortex count, loading and reading back at sizes around the
edges of their work splits (28 columns a warp, 8 warps a block, marches of a
few points, 256 points of a row), against the FP64 oracle.

Tolerances as for every comparison of the observables: 1e-12 relative in
complex double, 1e-5 in complex float (on the norms of the terms: a random
state's energies are dominated by the kinetic term, 1/h^2)."""
import numpy as np
import pytest

import oracle
from paper_1906_06327_gb300.rotgp import Solver

pytestmark = pytest.mark.gpu

SIZES = [(4, 4), (27, 9), (28, 8), (29, 17), (57, 300), (258, 31), (5, 4, 4), (29, 8, 19),
         (56, 9, 5), (86, 33, 40), (30, 258, 7)]
KW = dict(gamma=1.0, nu=1.2, g=40.0, omega=0.7)
NAMES = ("norm", "mu", "energy", "mu_c", "energy_c", "rms_x", "rms_y", "rms_z", "rms_r",
         "max_density", "mu4", "energy4")


def _state(n, seed):
    rng = np.random.default_rng(seed)
    shape = tuple(v + 1 for v in reversed(n))
    psi = rng.standard_normal(shape) + 1j * rng.standard_normal(shape)
    for ax in range(len(n)):
        sl = [slice(None)] * len(n)
        for e in (0, -1):
            sl[ax] = e
            psi[tuple(sl)] = 0
    return psi


@pytest.mark.parametrize("precision", ["fp32", "fp64"])
@pytest.mark.parametrize("n", SIZES)
def test_observables_at_split_edges(n, precision):
    h = (0.31, 0.27, 0.35)[:len(n)]
    kw = dict(KW, lam=1.3) if len(n) == 3 else KW
    psi = _state(n, 7).astype(np.complex64 if precision == "fp32" else np.complex128)
    s = Solver(n, h, dt=1e-3, precision=precision, **kw)
    s.set_psi(psi)
    got = s.get_psi(fp64=precision == "fp64")
    assert np.array_equal(got, psi)
    grid, phys = oracle.Grid(n, h), oracle.Phys(dt=1e-3, **kw)
    ref = oracle.observables(grid, phys, psi.astype(np.complex128))
    o = s.observables()
    tol = 1e-5 if precision == "fp32" else 1e-12
    for k in NAMES:
        assert abs(o[k] - ref[k]) <= tol * max(abs(ref[k]), 1.0), (k, o[k], ref[k])
    count = oracle.vortex_count(grid, psi.astype(np.complex128), fp32_decision=precision == "fp32")
    assert o["vortices"] == count
    # normalised on load: unit norm, the same shape of state
    s.set_psi(psi, normalise=True)
    want = psi / np.sqrt(ref["norm"])
    err = np.abs(s.get_psi() - want).max() / np.abs(want).max()
    assert err < (3e-7 if precision == "fp32" else 1e-15 * 4)
    assert abs(s.observables()["norm"] - 1) < (1e-6 if precision == "fp32" else 1e-13)
