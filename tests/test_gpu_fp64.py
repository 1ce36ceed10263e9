"""The plain FP64 pair kernel and the energy sums at the edges of their work splits, against the oracle.

Forces within 1e-12 of the sum of term magnitudes (as for every FP64 force); energies within 1e-13 of the oracle's
(n <= 4000 terms per sum, each within a few 2^-53, against a plain sum).
"""
import numpy as np
import pytest

import oracle
from paper_1406_6158_gb300 import ics

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def H():
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_1406_6158_gb300 import build, hybrid
    build.build()
    hybrid.load()
    return hybrid


def state(n, same=0):
    st = ics.plummer(n, 31 + n)
    for k in ("x", "y", "z"):
        st[k][:same] = 0.25
    return st


# slices of 4 sinks: groups below, at and above one slice, ragged last slices of every size, groups above
# 32 slices (the cap: rounds), and a leaf of coincident particles larger than n_crit with and without softening
@pytest.mark.parametrize("n,n_crit,same,eps", [(1, 64, 0, 0.01), (2, 1, 0, 0.01), (700, 1, 0, 0.01), (700, 4, 0, 0.01),
                                               (701, 5, 0, 0.01), (900, 128, 0, 0.01), (700, 8, 0, 0.01),
                                               (701, 9, 0, 0.01), (1500, 64, 0, 0.01), (1500, 300, 0, 0.01),
                                               (900, 16, 333, 0.01), (900, 16, 333, 0.0)])
def test_fp64_forces_at_the_splits_edges(H, n, n_crit, same, eps):
    st = state(n, same)
    P = H.Params(eps=eps, theta=0.6, R1=0.04, R2=0.08, precision=0, n_crit=n_crit, n_leaf=min(16, n_crit))
    ctx, s = H.Context(P), H.System(st, precision=0)
    ctx.hybrid_build_tree(s)
    ctx.hybrid_hard_force(s)
    ctx.hybrid_soft_force(s)
    out = s.numpy()
    T = oracle.Tree(out["x"], out["y"], out["z"], out["m"],
                    oracle.Params(eps=eps, theta=0.6, R1=0.04, R2=0.08, n_crit=n_crit, n_leaf=min(16, n_crit)))
    a_s, a_h, sc_s, sc_h = T.forces()
    # without softening the oracle has no value (0 / 0) for the coincident particles
    ok = np.isfinite(sc_s) & np.isfinite(sc_h)
    assert np.sum(~ok) == (same if eps == 0.0 else 0)
    floor = 1e-24 * np.max(sc_s[ok])   # a pair at r = R2 to the last bit: K ~ 1e-90 or 0

    def check(o):
        for d, k in enumerate("xyz"):
            assert np.all(np.abs(o["a%s_s" % k] - a_s[:, d])[ok] <= 1e-12 * sc_s[ok] + floor)
            assert np.all(np.abs(o["a%s_h" % k] - a_h[:, d])[ok] <= 1e-12 * sc_h[ok] + floor)
    check(out)
    # both forces in one launch (a step's first forces): the combined walk lists the same entries in another order
    s2, ctx2 = H.System(st, precision=0), H.Context(P)
    ctx2.hybrid_step(s2, 0)
    check(s2.numpy())


# the FP64 walk: every cell opened (more pending cells than the shared part of a warp's stack holds), none, leaves of
# 1 particle and leaves of 32 and more (offsets by ballots and by scan); leaves above 128 (moments by a whole warp)
@pytest.mark.parametrize("n,theta,n_leaf,same", [(6000, 0.0, 1, 0), (3000, 1e-3, 16, 0), (2500, 0.6, 31, 0),
                                                 (2500, 0.6, 64, 0), (2500, 5.0, 1, 0), (1500, 0.6, 16, 40),
                                                 (2500, 0.6, 64, 129), (2500, 0.6, 300, 0)])
def test_fp64_walk_at_its_edges(H, n, theta, n_leaf, same):
    st = state(n, same)
    kw = dict(eps=0.01, theta=theta, R1=0.04, R2=0.08, n_crit=64, n_leaf=n_leaf)
    ctx, s = H.Context(H.Params(precision=0, **kw)), H.System(st, precision=0)
    ctx.hybrid_step(s, 0)
    o = s.numpy()
    T = oracle.Tree(o["x"], o["y"], o["z"], o["m"], oracle.Params(**kw))
    a_s, a_h, sc_s, sc_h = T.forces()
    floor = 1e-24 * np.max(sc_s)
    for d, k in enumerate("xyz"):
        assert np.all(np.abs(o["a%s_s" % k] - a_s[:, d]) <= 1e-12 * sc_s + floor)
        assert np.all(np.abs(o["a%s_h" % k] - a_h[:, d]) <= 1e-12 * sc_h + floor)


@pytest.mark.parametrize("scale", [-328, -300, 300, 330])
def test_fp64_forces_scale_with_the_lengths(H, scale):
    # lengths times 2^scale: forces times 2^(-2 scale) (inside the seed's range, 2^-640 < r^2 < 2^640, bit for
    # bit; beyond it the fallback's roundings differ, a few 2^-53 per term)
    f = 2.0 ** scale
    st = state(800)
    res = []
    for g in (1.0, f):
        P = H.Params(eps=0.01 * g, theta=0.6, R1=0.04 * g, R2=0.08 * g, precision=0)
        s = H.System(dict(st, x=st["x"] * g, y=st["y"] * g, z=st["z"] * g), precision=0)
        ctx = H.Context(P)
        ctx.hybrid_build_tree(s)
        ctx.hybrid_soft_force(s)
        ctx.hybrid_hard_force(s)
        res.append((s.acc("s").cpu().numpy() * g * g, s.acc("h").cpu().numpy() * g * g))
    for a, b in zip(*res):
        assert np.all(np.isfinite(a)) and np.all(np.isfinite(b)) and np.any(b != 0.0)
        tol = 0.0 if abs(scale) <= 300 else 1e-13 * np.max(np.abs(a))
        assert np.max(np.abs(a - b)) <= tol


@pytest.mark.parametrize("n", [1, 2, 63, 64, 65, 255, 256, 257, 320, 1023, 4000])
def test_energy_at_the_tiles_edges(H, n):
    st = state(n)
    T0, W0 = oracle.energy(*[st[k] for k in ("x", "y", "z", "vx", "vy", "vz", "m")], G=0.7, eps=0.02)
    ctx, s = H.Context(H.Params(G=0.7, eps=0.02)), H.System(st, precision=1)
    T, W = ctx.hybrid_energy(s)
    Tn, Wn = H.hybrid_energy_noalloc(*[s.t[k] for k in H.System.FIELDS], 0.7, 0.02)
    for a, b in ((T, T0), (W, W0), (Tn, T0), (Wn, W0)):
        assert abs(a - b) <= 1e-13 * abs(b)
    assert (T, W) == ctx.hybrid_energy(s)


def test_energy_beyond_the_seeds_range(H):
    st = state(300)
    W0 = H.Context(H.Params(eps=0.0)).hybrid_energy(H.System(st))[1]
    for scale in (-460, 460):   # r^2 ~ 2^(2 scale): sqrt and division
        f = 2.0 ** scale
        s = H.System(dict(st, x=st["x"] * f, y=st["y"] * f, z=st["z"] * f))
        W = H.Context(H.Params(eps=0.0)).hybrid_energy(s)[1]
        assert abs(W * f - W0) <= 1e-13 * abs(W0)


# pairs alone, so that a force is one term: m / r^2 and the potential m / r, over binades, at both edges of [1, 4) and
# beyond the fixed-point range. A term is rounded when r^2 is made (2 units of 2^-53: exact for one coordinate, r^2
# itself 1), by x^-3/2 or x^-1/2 (2 units, by sqrt and division 9) and by products here and there (4): 2^-49 is 16
@pytest.mark.parametrize("E", [-330, -321, -320, -319, -40, -1, 0, 1, 2, 33, 318, 319, 320, 330])
def test_fp64_single_pairs(H, E):
    rng = np.random.default_rng(E + 1000)
    for r in list(2.0 ** rng.uniform(0, 1, 6)) + [1.0, np.nextafter(1.0, 2.0), np.nextafter(2.0, 1.0)]:
        r = float(np.ldexp(r, E))
        z = np.zeros(2)
        st = dict(x=np.array([0.0, r]), y=z, z=z, vx=z, vy=z, vz=z, m=np.array([1.0, 1.5]))
        ctx = H.Context(H.Params(eps=0.0, theta=0.5, R1=0.0, R2=0.0, precision=0))
        s = H.System(st, precision=0)
        T, W = ctx.hybrid_energy(s)
        assert abs(W * r + 1.5) <= 1.5 * 2.0 ** -49
        ctx.hybrid_build_tree(s)
        ctx.hybrid_soft_force(s)
        a = s.numpy()["ax_s"]
        for v, m in ((a[np.argmin(s.numpy()["x"])], 1.5), (-a[np.argmax(s.numpy()["x"])], 1.0)):
            assert abs(v * r * r - m) <= m * 2.0 ** -49
