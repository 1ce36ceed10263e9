"""Nodes and sink groups at the edges of the topology kernels' tiles and windows, bit for bit against the oracle."""
import numpy as np
import pytest

import oracle
from paper_1406_6158_gb300 import ics
from test_gpu_parity import H, check_tree, oparams  # noqa: F401

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


def tree_of(H, st, **kw):
    P = H.Params(eps=0.01, theta=0.6, R1=0.04, R2=0.08, **kw)
    ctx, s = H.Context(P), H.System(st, precision=P.precision)
    ctx.hybrid_build_tree(s)
    T = oracle.Tree(st["x"], st["y"], st["z"], st["m"], oparams(P))
    assert np.array_equal(s.numpy()["id"], T.perm)
    return T, ctx.tree(s.n)


# tiles of 1024 particles (the end of the batch is a position of its own), windows of n_leaf and n_crit, groups
# from the cells (n_crit <= 1024) and from the nodes (above)
@pytest.mark.parametrize("n", [1, 2, 1023, 1024, 1025, 2048, 5000])
@pytest.mark.parametrize("n_leaf,n_crit", [(1, 1), (16, 64), (16, 5), (3, 256), (40, 1024), (16, 1025), (7, 100000)])
def test_tiles_and_windows(H, n, n_leaf, n_crit):  # noqa: F811
    check_tree(*tree_of(H, ics.plummer(n, 77 + n), n_leaf=n_leaf, n_crit=n_crit, precision=1), 1)


@pytest.mark.parametrize("n_leaf,n_crit", [(16, 64), (300, 500), (2000, 64)])
def test_coincident_particles_across_tiles(H, n_leaf, n_crit):  # noqa: F811
    st = ics.plummer(4000, 5)
    for k in "xyz":
        st[k][500:1900] = 0.125      # 1400 particles in one cell of the finest level
        st[k][3000:3010] = -0.5
    check_tree(*tree_of(H, st, n_leaf=n_leaf, n_crit=n_crit, precision=0), 0)


def test_batch_boundaries(H):  # noqa: F811
    # systems that end inside, at and past a tile's end: each must get the tree it has alone
    sizes = [1024, 1, 1023, 3000, 2, 40]
    P = H.Params(eps=0.01, theta=0.6, R1=0.04, R2=0.08, precision=0)
    states = [ics.plummer(n, 200 + n) for n in sizes]
    systems = [H.System(st, precision=0) for st in states]
    H.Context(P).hybrid_step_batched(systems, 0)
    for st, s in zip(states, systems):
        alone = H.System(st, precision=0)
        H.Context(P).hybrid_step(alone, 0)
        a, b = alone.numpy(), s.numpy()
        for k in a:
            assert np.array_equal(a[k], b[k]), k


def test_search_for_the_farthest_particle(H):  # noqa: F811
    # above 2^20 particles b_max of the larger cells is searched for: uneven clumps, coincident particles, a lattice
    # (many particles at the same distance) and outliers, against the oracle's largest distance
    n = (1 << 20) + 3000
    st = ics.plummer(n, 12)
    rng = np.random.default_rng(5)
    for k, d in enumerate("xyz"):
        st[d][:400000] = 0.3 + 0.01 * rng.standard_normal(400000)
        st[d][400000:402000] = 0.75
        st[d][402000:410000] = (np.arange(8000) // 20 ** k % 20) / 16.0 - 3.0
    st["x"][500000] = 60.0
    check_tree(*tree_of(H, st, n_leaf=16, n_crit=256, precision=1), 1)


# group boxes: sub-warps of eight lanes, several groups after one another on large systems, and groups that take the
# whole warp (more than 1024 particles: of one level-21 cell, or by n_crit). Exact: minimum and maximum of the members.
@pytest.mark.parametrize("n,n_crit,same", [(1, 64, 0), (7, 1, 0), (1000, 5, 0), (5000, 64, 1024), (5000, 64, 1025),
                                           (9000, 2000, 0), (400000, 1, 0)])
def test_group_boxes_are_the_members_bounds(H, n, n_crit, same):  # noqa: F811
    st = ics.plummer(n, 5)
    for k in ("x", "y", "z"):
        st[k][:same] = 0.125
    ctx, s = H.Context(H.Params(n_crit=n_crit, n_leaf=min(16, n_crit))), H.System(st)
    ctx.hybrid_build_tree(s)
    t, o = ctx.tree(n), s.numpy()
    first = t["first"][t["gnode"]]
    for d, k in enumerate("xyz"):
        assert np.array_equal(t["glo"][:, d], np.minimum.reduceat(o[k], first))
        assert np.array_equal(t["ghi"][:, d], np.maximum.reduceat(o[k], first))
