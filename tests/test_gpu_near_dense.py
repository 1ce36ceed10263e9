"""Near forces of states with many pairs within R2, next to ones with few, against the oracle.

As for every FP32 force: soft and hard within 1e-5 relative at the 99th percentile, hard forces exactly zero where no
neighbour lies within R2.
"""
import numpy as np
import pytest

import oracle
from paper_1406_6158_gb300 import ics
from test_gpu_near import check
from test_gpu_parity import H, oparams, sampled_lists_match  # noqa: F401

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


def clumped(n, m, radius, seed):
    st = ics.plummer(n, seed)
    rng = np.random.default_rng(seed)
    for d in "xyz":
        st[d][:m] = 0.2 + radius * rng.standard_normal(m)
    return st


# groups of a few sinks (many copies of them in a warp) to several blocks of them; a clump well inside R2 (every pair
# within), about as large (about half), and none; odd numbers of sources
@pytest.mark.parametrize("n_crit", [1, 2, 3, 5, 11, 20, 33, 64, 100, 300])
@pytest.mark.parametrize("m,radius", [(1501, 0.004), (1500, 0.05), (0, 0.0)])
def test_forces_of_a_clump(H, n_crit, m, radius):  # noqa: F811
    n = 4001
    st = clumped(n, m, radius, 3 + n_crit)
    P = H.Params(eps=0.01, theta=0.5, R1=0.03, R2=0.08, n_crit=n_crit, n_leaf=min(16, n_crit), precision=1)
    ctx, s = H.Context(P), H.System(st, precision=1)
    ctx.hybrid_build_tree(s)
    ctx.hybrid_soft_force(s)
    ctx.hybrid_hard_force(s)
    out = s.numpy()
    T = oracle.Tree(out["x"], out["y"], out["z"], out["m"], oparams(P))
    check(out, T)
    both = H.System(st, precision=1)
    ctx.hybrid_step(both, 0)
    check(both.numpy(), T)


@pytest.mark.parametrize("eps", [0.0, 0.002])
def test_forces_and_lists_of_a_batch_with_and_without_clumps(H, eps):  # noqa: F811
    states = [clumped(2500, 900, 0.003, 1), ics.plummer(1, 2), clumped(30, 30, 0.001, 3), ics.plummer(3000, 4)]
    P = H.Params(eps=eps, theta=0.6, R1=0.02, R2=0.05, precision=1)
    systems = [H.System(st, precision=1) for st in states]
    H.Context(P).hybrid_step_batched(systems, 0)
    for st, s in zip(states, systems):
        out = s.numpy()
        T = oracle.Tree(out["x"], out["y"], out["z"], out["m"], oparams(P))
        check(out, T)
        ctx, alone = H.Context(P), H.System(st, precision=1)
        ctx.hybrid_build_tree(alone)
        ctx.hybrid_hard_force(alone)
        sel = np.arange(T.ng)
        ol = T.walk(sel, mode=2)
        flips = sampled_lists_match(T, ctx.lists(T.ng, sel), ol, sel)
        assert flips <= 1e-4 * sum(len(b[2]) for b in ol) + 1
