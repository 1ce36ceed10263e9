"""Near forces in units where R2 is a very large number (metres, centimetres): the same forces, scaled."""
import numpy as np
import pytest

from test_gpu_parity import H  # noqa: F401

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("n,n_crit", [(700, 1), (2001, 33), (5003, 64), (3000, 500)])
@pytest.mark.parametrize("both", [False, True], ids=["hard", "soft_and_hard"])
def test_hard_forces_scale_with_the_units(H, n, n_crit, both):  # noqa: F811
    # lengths times 2^63 (9.2e18) and masses times 2^100: accelerations times 2^(100 - 126) exactly, since every FP32
    # value of a near pair stays a normal number. R2 = 0.17 * 2^63 = 1.6e18. The sums are in no fixed order: 1e-5.
    rng = np.random.default_rng(n)
    st = {k: rng.uniform(0.0, 1.0, n) for k in "xyz"}
    st.update({k: np.zeros(n) for k in ("vx", "vy", "vz")})
    st["m"] = np.full(n, 1.0 / n)
    res = []
    for L, M in ((0, 0), (63, 100)):
        t = {k: v * 2.0 ** (L if k in "xyz" else M if k == "m" else 0) for k, v in st.items()}
        P = H.Params(eps=0.01 * 2.0 ** L, theta=0.6, R1=0.08 * 2.0 ** L, R2=0.17 * 2.0 ** L, n_crit=n_crit,
                     n_leaf=min(16, n_crit), precision=1)
        ctx, s = H.Context(P), H.System(t, precision=1)
        if both:
            ctx.hybrid_step(s, 0)
        else:
            ctx.hybrid_build_tree(s)
            ctx.hybrid_hard_force(s)
        o = s.numpy()
        a = np.stack([o["a%s_h" % d] for d in "xyz"], 1).astype(np.float64)
        res.append(a[np.argsort(o["id"])] * 2.0 ** (2 * L - M))
    a, b = res
    assert np.abs(a).max() > 0.0
    assert np.max(np.abs(a - b)) <= 1e-5 * np.abs(a).max()
