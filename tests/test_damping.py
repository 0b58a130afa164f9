"""Imaginary-time steps in complex float whose H1 factors are far below 1: every
point to its own relative accuracy, in each form of the default plan (the on-chip
2D stepper, tiles on odd rows and with long halos, the sweeps), against the oracle.

Tolerance, relative to the point: the exponent u is rounded some four times
(4 |u| 2^-24) and e^u is right to 2 + 1.2 |u| units of 2^-23; the sweeps, whose
neighbours weigh as much as the point itself, and the scale add ten roundings."""
import numpy as np
import pytest

import oracle
from paper_1906_06327_gb300.rotgp import Solver

pytestmark = pytest.mark.gpu

DEEP = 16.0  # about the largest -u: V Delta in the corners


@pytest.mark.parametrize("n,kappa", [((65, 48), 0.02), ((64, 48), 0.1), ((65, 48, 20), 0.02),
                                     ((90, 80), 0.6),
                                     ((40, 32, 20), 0.02)])
def test_points_keep_their_relative_accuracy(n, kappa):
    h = (0.4,) * len(n)
    dt = 4.0 * kappa * h[0] ** 2
    r2 = sum((0.5 * h[0] * v) ** 2 for v in n)
    w = float(np.sqrt(2.0 * DEEP / (dt * r2)))  # the trap frequency of that depth
    kw = dict(gamma=w, nu=w, lam=w, g=10.0, omega=0.02, dt=dt)
    rng = np.random.default_rng(1)
    psi = np.zeros(tuple(v + 1 for v in reversed(n)), np.complex128)
    core = tuple(slice(1, -1) for _ in n)
    psi[core] = rng.normal(size=psi[core].shape) + 1j * rng.normal(size=psi[core].shape)
    grid = oracle.Grid(n, h)
    psi = (psi / np.sqrt(oracle.norm(grid, psi))).astype(np.complex64)
    # neighbours within one step of each other, so that a point's own
    # rounding is what shows
    ref, _ = oracle.steps(grid, oracle.Phys(**kw), psi.astype(np.complex128), 1, True)
    s = Solver(n, h, **kw)
    s.set_psi(psi)
    s.step_imag(1)
    got = s.get_psi()
    near = np.abs(ref)
    for ax in range(ref.ndim):  # a point and its neighbours: what a sweep mixes
        near = np.maximum(near, np.maximum(np.roll(near, 1, ax), np.roll(near, -1, ax)))
    err = (np.abs(got - ref) / np.where(near > 0, near, 1)).max()
    assert err < 4 * DEEP * 2.0**-24 + (2 + 1.2 * DEEP) * 2.0**-23 + 10 * 2.0**-24, err
