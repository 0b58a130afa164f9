"""Graphs of several 2D instances: many small ones take their sweeps side by side, a
few take blocks of steps over the whole chip one after another.

Tolerance where forms differ: 4 x 6e-8 per step and form in complex float, 2e-15
in complex double, added up linearly (tests/test_resident.py,
tests/test_double_steps.py)."""
import time

import numpy as np
import pytest

from paper_1906_06327_gb300.rotgp import Batch, Solver

pytestmark = pytest.mark.gpu

KW = dict(gamma=1.0, nu=1.05, g=60.0, omega=0.6, dt=1e-3)


def _specs(n, count):
    return [dict(n=n, h=(12.0 / n[0], 12.0 / n[1]), **dict(KW, g=60.0 + i)) for i in range(count)]


def _single(spec, i, precision, form):
    kw = {k: v for k, v in spec.items() if k not in ("n", "h")}
    s = Solver(spec["n"], spec["h"], precision=precision, **kw)
    for ax in range(2 if form else 0):
        s.set_solver(ax, form)
    s.init_analytic(1, seed=i)
    s.step_imag(6)
    s.step_imag(5)
    s.step_real(4)
    return s.get_psi()


# (grid, instances, precision, mode, the form that single contexts ask for to give
# the same bits: "" the default, None no such form)
CASES = [((64, 48), 16, "fp32", "graph", "thomas"), ((64, 48), 16, "fp32", "direct", ""),
         ((64, 48), 2, "fp32", "graph", ""), ((128, 128), 12, "fp32", "graph", "thomas"),
         ((65, 48), 16, "fp32", "graph", None), ((64, 48), 12, "fp64", "graph", None)]


@pytest.mark.parametrize("n,count,precision,mode,form", CASES)
def test_matches_single_contexts(n, count, precision, mode, form):
    specs = _specs(n, count)
    b = Batch(specs, precision=precision)
    for i, s in enumerate(b.instances):
        s.init_analytic(1, seed=i)
    b.step_imag(6, mode=mode)
    b.step_imag(5, mode=mode)
    b.step_real(4, mode=mode)
    b.sync()
    for i in (0, 1, count - 1):
        got, want = b.instances[i].get_psi(), _single(specs[i], i, precision, form)
        if form is not None:
            assert np.array_equal(got, want), i
        else:
            per = 2 * 4 * 6e-8 if precision == "fp32" else 2e-15
            assert np.linalg.norm(got - want) < per * 15 * np.linalg.norm(want), i
    b.close()


@pytest.mark.parametrize("n,count,precision", [((128, 128), 32, "fp32"), ((64, 64), 32, "fp64")])
def test_a_graph_of_many_is_not_one_after_another(n, count, precision):
    """Less than the time of as many direct launches, which run in turn."""
    b = Batch(_specs(n, count), precision=precision)
    for i, s in enumerate(b.instances):
        s.init_analytic(1, seed=i)
    best = {}
    for mode in ("direct", "graph"):
        for _ in range(4):
            b.step_imag(50, mode=mode)
        b.sync()
        for _ in range(3):
            t = time.perf_counter()
            b.step_imag(50, mode=mode)
            b.sync()
            best[mode] = min(best.get(mode, 1e9), time.perf_counter() - t)
    b.close()
    assert best["graph"] < 0.7 * best["direct"], best


@pytest.mark.parametrize("mode", ["graph", "direct", "persistent"])
@pytest.mark.parametrize("precision", ["fp32", "fp64"])
def test_instances_follow_the_batch(mode, precision):
    """An instance read or stepped by itself right after a block of batch steps, with
    nothing waited for in between."""
    specs = _specs((128, 96), 6)
    got = []
    for wait in (True, False):
        b = Batch(specs, precision=precision)
        for i, s in enumerate(b.instances):
            s.init_analytic(1, seed=i)
        for _ in range(3):
            b.step_imag(150, mode=mode)
            if wait:
                b.sync()
        first = b.instances[5].get_psi()
        b.instances[4].step_real(3)
        b.step_imag(150, mode=mode)
        if wait:
            b.sync()
        b.instances[3].set_omega(0.4)
        b.instances[3].step_imag(4)
        got.append([first] + [s.get_psi() for s in b.instances])
        b.close()
    for x, y in zip(*got):
        assert np.array_equal(x, y)
