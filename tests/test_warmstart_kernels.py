"""The learned start's convolutions at the sizes where their tiles are ragged
(planes of 2 to 112 points a side, odd batches, more runs of tiles than slots
of partial sums)."""
import numpy as np
import pytest

from oracle import warmstart_ref as ref

pytestmark = pytest.mark.gpu


def _bf16(a):
    u = np.ascontiguousarray(a, dtype=np.float32).view(np.uint32)
    r = (u + 0x7FFF + ((u >> 16) & 1)) & 0xFFFF0000
    return r.astype(np.uint32).view(np.float32)


def _inputs(G, n, seed):
    rng = np.random.default_rng(seed)
    p = _bf16(ref.init_params(3).astype(np.float32) + 0.02 * rng.normal(size=ref.n_params()))
    x = _bf16(rng.normal(size=(n, G, G, ref.CIN)).astype(np.float32))
    return p, x, rng.normal(size=(n, G, G, 2)).astype(np.float32)


@pytest.mark.parametrize("G,n", [(16, 3), (48, 1)])
def test_gradients_match_fp64_reference(G, n):
    # activations are rounded to bfloat16 (2^-9) in every layer: the bounds of
    # the 32 x 32 comparison in test_warmstart.py
    from paper_1906_06327_gb300.rotgp import WarmStart
    p, x, t = _inputs(G, n, 11)
    ws = WarmStart(G, max_batch=n)
    ws.set_params(p)
    loss, g = ws.gradients(x, t)
    loss_ref, g_ref = ref.gradients(p.astype(np.float64), x.astype(np.float64), t.astype(np.float64))
    assert abs(loss - loss_ref) <= 1e-2 * loss_ref
    off = 0
    for shape in ref.param_shapes():
        k = int(np.prod(shape))
        a, b = g[off:off + k].astype(np.float64), g_ref[off:off + k]
        off += k
        assert np.linalg.norm(a - b) <= 6e-2 * np.linalg.norm(b), shape


@pytest.mark.parametrize("G,n", [(16, 131), (112, 5), (128, 17)])
def test_copies_of_a_run_share_its_gradient(G, n):
    # n copies of one run have its loss and gradient, summed over other blocks
    # and slots: a few thousand float additions (6e-8 each, random signs)
    from paper_1906_06327_gb300.rotgp import WarmStart
    p, x, t = _inputs(G, 1, 12)
    ws = WarmStart(G, max_batch=n)
    ws.set_params(p)
    loss, g = ws.gradients(x, t)
    many, gn = ws.gradients(np.repeat(x, n, axis=0), np.repeat(t, n, axis=0))
    assert abs(many - loss) <= 1e-6 * loss
    assert np.linalg.norm(gn - g) <= 2e-5 * np.linalg.norm(g)
    # and the same every time
    assert np.array_equal(gn, ws.gradients(np.repeat(x, n, axis=0), np.repeat(t, n, axis=0))[1])
