"""The builds' kernels where their form changes with the size of the batch: tiles of 256, 512 and 1024 positions, counts
added up by every block or scanned, bucket counts added up or scanned."""
import math

import numpy as np
import pytest

import oracle
from paper_1406_6158_gb300 import ics
from test_gpu_batch_memory import batch
from test_gpu_parity import H, check_tree, keyed_order, oparams, set_positions  # noqa: F401

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


# the end of the batch is a position of its own: 256 particles are two tiles. 320 tiles of 256 hold 81919 particles, 320
# of 512 163839, 320 of 1024 327679; above, the counts of the tiles are scanned
@pytest.mark.parametrize("n", [255, 256, 257, 511, 512, 81919, 81920, 131072, 163839, 163840, 327679, 327680])
@pytest.mark.parametrize("prec", [0, 1])
def test_tree_where_the_tiles_change(H, n, prec):  # noqa: F811
    st = ics.plummer(n, 8)
    P = H.Params(eps=0.01, theta=0.6, R1=0.04, R2=0.08, n_leaf=16, n_crit=64, precision=prec)
    ctx, s = H.Context(P), H.System(st, precision=prec)
    ctx.hybrid_build_tree(s)
    T = oracle.Tree(st["x"], st["y"], st["z"], st["m"], oparams(P))
    assert np.array_equal(s.numpy()["id"], T.perm)
    G = ctx.tree(n)
    if prec == 1:
        check_tree(T, G, 1)
        return
    # the nodes and groups bit for bit. The oracle adds a cell's particles one after another: its root mass is off by 1.5e-12
    # at 81920, so masses are held against the exact sums of their particles instead. Chunks of at most 128 in eight lanes,
    # then at most 21 levels of up to eight children: under 16 + 3 + 21 * 3 roundings of 2^-53 each, 1e-14
    for f in ("key", "level", "first", "count", "child", "nchild", "parent", "gnode", "glo", "ghi"):
        assert np.array_equal(G[f], getattr(T, f)), f
    m = s.numpy()["m"]
    for c in np.concatenate([np.arange(min(T.nn, 9)), np.random.default_rng(n).integers(0, T.nn, 200)]):
        exact = math.fsum(m[G["first"][c]:G["first"][c] + G["count"][c]])
        assert abs(G["moments"][c, 0] - exact) <= 1e-14 * exact


@pytest.mark.parametrize("sizes", [[40000, 41919, 1], [40000, 41919], [1, 163838], [163838, 1, 1], [327000, 679, 1]])
def test_batches_where_the_tiles_change(H, sizes):  # noqa: F811
    P = H.Params(eps=0.01, theta=0.6, R1=0.02, R2=0.04, precision=0)
    states = [ics.plummer(n, 60 + n) for n in sizes]
    systems = [H.System(st, precision=0) for st in states]
    H.Context(P).hybrid_step_batched(systems, 0)
    for st, s in zip(states, systems):
        alone = H.System(st, precision=0)
        H.Context(P).hybrid_step(alone, 0)
        a, b = alone.numpy(), s.numpy()
        for k in a:
            assert np.array_equal(a[k], b[k]), k


# 4096 buckets of 224 are 917504 particles: above, the sort reads scanned counts
@pytest.mark.parametrize("n", [917504, 917505, (1 << 20) + 3000])
def test_sample_sort_where_the_counts_are_scanned(H, n):  # noqa: F811
    st = ics.plummer(n, 14)
    st = {k: v[keyed_order(st)].copy() for k, v in st.items()}
    ctx, s = H.Context(H.Params(eps=0.01, precision=1)), H.System(st, precision=1)
    ctx.hybrid_build_tree(s)
    f0 = ctx.hybrid_sort_fallbacks()
    for d in "xyz":
        st[d] = st[d] + 1e-3 * st["v" + d]
    set_positions(s, st)
    ctx.hybrid_build_tree(s)
    assert np.array_equal(s.numpy()["id"], keyed_order(st))
    assert ctx.hybrid_sort_fallbacks() == f0


def test_new_small_systems_where_the_counts_are_scanned(H):  # noqa: F811
    # 2000 new systems of 600 particles, 6000 buckets: each sorted with splitters of its own, beside the scanned counts
    S, n = 2000, 600
    t, arr = batch(H, S, n)
    old = {k: t[k].cpu().numpy().copy() for k in "xyz"}
    ctx = H.Context(H.Params(eps=0.05, theta=0.5, R1=0.1, R2=0.2))
    assert ctx.L.hybrid_step_batched(ctx.h, arr, S, 0) == 0
    assert ctx.hybrid_sort_fallbacks() == 0
    new = {k: t[k].cpu().numpy() for k in "xyz"}
    for s in range(0, S, 37):
        cut = slice(s * n, (s + 1) * n)
        order = keyed_order({k: v[cut] for k, v in old.items()})
        for k in "xyz":
            assert np.array_equal(new[k][cut], old[k][cut][order])


def test_overflow_of_a_large_system(H):  # noqa: F811
    # splitters that do not fit the state, from their definition: every 224-th of the sorted composites (key, position) of
    # the build before. A bucket of the new state's composites with more than 512 sends the build to the radix sort.
    n = 100000
    st = ics.plummer(n, 91)
    st = {k: v[keyed_order(st)].copy() for k, v in st.items()}
    cube = {k: v.copy() for k, v in st.items()}
    rng = np.random.default_rng(4)
    for d in "xyz":
        cube[d] = rng.uniform(-1.0, 1.0, n)

    def composites(q):
        lo, L = oracle.root_box(q["x"], q["y"], q["z"])
        return oracle.morton_keys(q["x"], q["y"], q["z"], lo, L).astype(object) * n + np.arange(n)
    split = composites(st)[224::224]
    assert np.all(split[1:] > split[:-1])
    ctx, s = H.Context(H.Params(eps=0.01)), H.System(st)
    ctx.hybrid_build_tree(s)
    f0 = ctx.hybrid_sort_fallbacks()
    assert np.bincount(np.searchsorted(split, composites(cube), side="right").astype(np.int64)).max() > 512
    set_positions(s, cube)
    ctx.hybrid_build_tree(s)
    assert ctx.hybrid_sort_fallbacks() == f0 + 1
    assert np.array_equal(s.numpy()["id"], keyed_order(cube))
    ctx.hybrid_build_tree(s)   # and the build after it takes the sample sort again
    assert ctx.hybrid_sort_fallbacks() == f0 + 1
