"""The sample sort at the edges of its buckets: the stable order of the keys, whatever the buckets hold."""
import numpy as np
import pytest

from paper_1406_6158_gb300 import ics
from test_gpu_parity import H, keyed_order, set_positions  # noqa: F401

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


def built(H, n, seed):
    st = ics.plummer(n, seed)
    st = {k: v[keyed_order(st)].copy() for k, v in st.items()}
    ctx, s = H.Context(H.Params(eps=0.01, precision=1)), H.System(st, precision=1)
    ctx.hybrid_build_tree(s)
    return st, ctx, s


# buckets of 224 positions: one bucket, full last buckets, a last bucket of one, many
@pytest.mark.parametrize("n", [1, 2, 223, 224, 225, 448, 449, 512, 513, 4096, 20011])
def test_order_after_a_drift(H, n):  # noqa: F811
    st, ctx, s = built(H, n, 300 + n)
    f0 = ctx.hybrid_sort_fallbacks()
    for k, d in enumerate("xyz"):
        st[d] = st[d] + 2e-3 * st["v" + d]
    set_positions(s, st)
    ctx.hybrid_build_tree(s)
    assert np.array_equal(s.numpy()["id"], keyed_order(st))
    assert ctx.hybrid_sort_fallbacks() == f0


# m particles from all over the array put on one point: a bucket of 224 + m keys, below and above 256 (8 or 16 keys
# a lane) and above 512 (the radix sort)
@pytest.mark.parametrize("m,falls_back", [(20, False), (33, False), (200, False), (400, True)])
def test_crowded_bucket(H, m, falls_back):  # noqa: F811
    n = 30000
    st, ctx, s = built(H, n, 7)
    f0 = ctx.hybrid_sort_fallbacks()
    pick = np.random.default_rng(m).choice(n, m, replace=False)
    at = 15100   # a particle well inside bucket 67 (positions 15008 to 15231)
    for d in "xyz":
        st[d][pick] = st[d][at]
    set_positions(s, st)
    ctx.hybrid_build_tree(s)
    assert np.array_equal(s.numpy()["id"], keyed_order(st))
    assert (ctx.hybrid_sort_fallbacks() > f0) == falls_back
    out = s.numpy()
    ctx.hybrid_build_tree(s)   # and again, from the new order
    assert np.array_equal(s.numpy()["x"], out["x"])


def test_batch_with_other_sizes_than_the_last(H):  # noqa: F811
    # splitters of another layout: out of order for this batch, right all the same
    P = H.Params(eps=0.01, precision=0)
    ctx = H.Context(P)
    for sizes in ([5000], [700, 1, 3000, 224, 513], [2000, 2000]):
        states = [ics.plummer(n, 900 + n) for n in sizes]
        systems = [H.System(st, precision=0) for st in states]
        ctx.hybrid_step_batched(systems, 0)
        ctx.hybrid_step_batched(systems, 0)
        for st, s in zip(states, systems):
            assert np.array_equal(s.numpy()["id"], keyed_order(st))
