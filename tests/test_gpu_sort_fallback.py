"""What a call does after a bucket of the sample sort has overflowed."""
import numpy as np
import pytest

from paper_1406_6158_gb300 import ics
from test_gpu_parity import H, keyed_order, set_positions  # noqa: F401

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

FIELDS = ("x", "y", "z", "vx", "vy", "vz", "ax_s", "ay_s", "az_s", "ax_h", "ay_h", "az_h", "id")


def sorted_plummer(n, seed):
    st = ics.plummer(n, seed)
    return {k: v[keyed_order(st)].copy() for k, v in st.items()}


@pytest.mark.parametrize("graphs", [False, True], ids=["eager", "graphs"])
def test_radix_sort_for_one_build_only(H, graphs):  # noqa: F811
    # 900 particles from all over put close together: the step's first build falls back to the radix sort, the four
    # after it do not (the radix sort takes eight launches more). The state is that of a step from the same state in
    # key order, bit for bit in the FP64 form.
    n = 9000
    st = sorted_plummer(n, 3)
    P = H.Params(eps=0.02, theta=0.6, R1=0.05, R2=0.1, precision=0, dt_soft=1 / 256)
    ctx = H.Context(P, torch.cuda.Stream() if graphs else None)
    s = H.System(st, precision=0)
    torch.cuda.synchronize()
    ctx.hybrid_build_tree(s)
    rng = np.random.default_rng(1)
    pick = rng.choice(n, 900, replace=False)
    for d in "xyz":
        st[d][pick] = 0.3 + 0.02 * rng.standard_normal(900)
    order = keyed_order(st)
    st = {k: v.copy() for k, v in st.items()}
    set_positions(s, st)
    s.t["id"].copy_(torch.arange(n, dtype=torch.int32))
    torch.cuda.synchronize()
    f0, l0 = ctx.hybrid_sort_fallbacks(), ctx.hybrid_launch_count()
    ctx.hybrid_step(s, 1)
    torch.cuda.synchronize()
    assert ctx.hybrid_sort_fallbacks() == f0 + 1
    launches = ctx.hybrid_launch_count() - l0

    other = H.Context(P, torch.cuda.Stream() if graphs else None)
    q = H.System({k: st[k][order] for k in H.System.FIELDS}, precision=0)
    torch.cuda.synchronize()
    other.hybrid_build_tree(q)
    f1, l1 = other.hybrid_sort_fallbacks(), other.hybrid_launch_count()
    other.hybrid_step(q, 1)
    torch.cuda.synchronize()
    assert other.hybrid_sort_fallbacks() == f1
    plain = other.hybrid_launch_count() - l1
    a, b = s.numpy(), q.numpy()
    b["id"] = order[b["id"]].astype(np.int32)
    for k in FIELDS:
        assert np.array_equal(a[k], b[k]), k
    assert plain < launches <= 2 * plain + 8


# a system of up to 19 buckets of 224 particles that is far from key order (a new state, another system's splitters) is
# sorted with splitters of its own, with no fallback; the sizes around one, two and eight regions of 512 keys, and the last
@pytest.mark.parametrize("n", [513, 600, 1023, 1024, 1025, 2048, 4095, 4096, 4097, 4255, 4256])
@pytest.mark.parametrize("prec", [0, 1])
def test_small_new_systems_take_no_fallback(H, n, prec):  # noqa: F811
    ctx = H.Context(H.Params(eps=0.01, precision=prec))
    for seed in (1, 2):
        st = ics.plummer(n, 700 + n + seed)
        rng = np.random.default_rng(seed)
        pick = rng.choice(n, n // 3, replace=False)   # ties: equal keys keep their order
        for d in "xyz":
            st[d][pick] = st[d][pick[np.arange(len(pick)) % 7]]
        s = H.System(st, precision=prec)
        ctx.hybrid_build_tree(s)
        assert np.array_equal(s.numpy()["id"], keyed_order(st))
        assert ctx.hybrid_sort_fallbacks() == 0


def test_small_new_systems_in_a_batch(H):  # noqa: F811
    # new small systems beside ones in key order: each gets its stable order, without a fallback; and beside a new large
    # one, with one
    P = H.Params(eps=0.01, precision=0)
    ctx = H.Context(P)
    sizes = [600, 100, 3000, 1, 4256, 513]
    states = [ics.plummer(n, 40 + n) for n in sizes]
    for k in (1, 3):
        states[k] = sorted_plummer(sizes[k], 40 + sizes[k])
    for st in (states, states[::-1]):
        systems = [H.System(q, precision=0) for q in st]
        ctx.hybrid_step_batched(systems, 0)
        for q, s in zip(st, systems):
            assert np.array_equal(s.numpy()["id"], keyed_order(q))
        assert ctx.hybrid_sort_fallbacks() == 0
    big = ics.plummer(9000, 3)
    systems = [H.System(q, precision=0) for q in states + [big]]
    ctx.hybrid_step_batched(systems, 0)
    for q, s in zip(states + [big], systems):
        assert np.array_equal(s.numpy()["id"], keyed_order(q))
    assert ctx.hybrid_sort_fallbacks() == 1


def test_small_system_whose_own_splitters_overflow(H):  # noqa: F811
    # half of the particles on one point, none of them among the 256 that the splitters are made of (every 16th): their
    # bucket overflows again, and the build is repeated with the radix sort
    n = 4096
    st = ics.plummer(n, 12)
    pick = np.flatnonzero(np.arange(n) % 16 > 7)
    for d in "xyz":
        st[d][pick] = 0.3
    ctx, s = H.Context(H.Params(eps=0.01)), H.System(st)
    ctx.hybrid_build_tree(s)
    assert np.array_equal(s.numpy()["id"], keyed_order(st))
    assert ctx.hybrid_sort_fallbacks() == 1
