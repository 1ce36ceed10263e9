"""A reused-lists drift that ends with a particle too far from its place at the last build is still a whole drift.

The step then goes on after that drift with rebuilt lists, so every particle must have had its kicks and its drift,
also where the launch has more blocks than the GPU holds at once.
"""
import numpy as np
import pytest

from paper_1406_6158_gb300 import ics
from test_gpu_parity import H  # noqa: F401

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("n", [1, 300, 300011, 1000003])
@pytest.mark.parametrize("graphs", [False, True], ids=["eager", "graphs"])
def test_exceeded_skin_leaves_the_drift_whole(H, n, graphs):  # noqa: F811
    # A skin of 1e-7 is exceeded by the first drift of every step. Without a skin the step rebuilds every time: the same
    # scheme, with lists that differ in the skin's 1e-7. A launch that skips a particle loses its drift, v dt_hard at
    # least. The two runs themselves differ by the forces' error: accelerations are below 3 here (mean field 0.39, an
    # encounter 0.39 m / eps^2), and the tree's error is below a hundredth of that, so over two steps positions differ
    # by at most 0.5 * 0.03 * (2 / 2048)^2 = 1.5e-8: under a hundredth of the drift of a particle faster than 0.05
    # (0.01 * 0.05 / 2048 / 4 = 6e-8).
    st = ics.plummer(n, 4)
    res = []
    for skin in (0.0, 1e-7):
        eps = 1 / (4 * n ** (1 / 3))
        P = H.Params(eps=eps, theta=0.5, R1=2 * eps, R2=4 * eps, dt_soft=1 / 2048, n_hard=4, skin=skin)
        ctx = H.Context(P, torch.cuda.Stream() if graphs else None)
        s = H.System(st, precision=1)
        torch.cuda.synchronize()
        ctx.hybrid_step(s, 0)
        ctx.hybrid_step(s, 1)
        ctx.hybrid_step(s, 1)
        out = s.numpy()
        res.append({k: out[k][np.argsort(out["id"])] for k in H.System.FIELDS})
        ctx.close()
    a, b = res
    v = np.sqrt(a["vx"] ** 2 + a["vy"] ** 2 + a["vz"] ** 2)
    d = np.sqrt(sum((a[k] - b[k]) ** 2 for k in "xyz"))
    fast = v > 0.05
    assert np.all(d[fast] <= 0.01 * v[fast] * P.dt_soft / P.n_hard)


@pytest.mark.parametrize("graphs", [False, True], ids=["eager", "graphs"])
@pytest.mark.parametrize("other", [100, 3000, 250000])
def test_energy_of_another_system_between_steps(H, graphs, other):  # noqa: F811
    # the energy of a larger system makes the context's buffers anew: the lists of the last step are gone then, and the
    # next step must not take them up. Positions follow the steps without it as far as lists in another order may
    # differ (FP32 forces: 1e-8, as in the comparison of reused lists with the oracle)
    n = 3000
    st, big = ics.plummer(n, 9), ics.plummer(other, 10)
    res = []
    for between in (False, True):
        P = H.Params(eps=1 / 64, theta=0.0, R1=4 / 64, R2=8 / 64, dt_soft=1 / 128, n_hard=4, skin=0.05)
        ctx = H.Context(P, torch.cuda.Stream() if graphs else None)
        s, o = H.System(st, precision=1), H.System(big, precision=1)
        torch.cuda.synchronize()
        for _ in range(3):
            ctx.hybrid_step(s, 1)
            if between:
                ctx.hybrid_energy(o)
        out = s.numpy()
        res.append({k: out[k][np.argsort(out["id"])] for k in H.System.FIELDS})
        ctx.close()
    for k in "xyz":
        assert np.max(np.abs(res[0][k] - res[1][k])) <= 1e-8, k
