"""Group sizes up to the largest that n_crit can name: every system is then one group, whatever the exact value."""
import numpy as np
import pytest

from paper_1406_6158_gb300 import ics
from test_gpu_parity import H  # noqa: F401

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("prec", [0, 1])
@pytest.mark.parametrize("n_crit", [1200, 2 ** 31 - 4, 2 ** 31 - 3, 2 ** 31 - 1])
def test_one_group_whatever_n_crit_above_n(H, prec, n_crit):  # noqa: F811
    # the lists, and so in the FP64 form every bit, are those of n_crit = n; FP32 sums are in no fixed order: 1e-5
    n = 1200
    st = ics.plummer(n, 6)
    res = []
    for crit in (n, n_crit):
        P = H.Params(eps=0.01, theta=0.6, R1=0.1, R2=0.2, n_crit=crit, precision=prec)
        ctx, s = H.Context(P), H.System(st, precision=prec)
        ctx.hybrid_step(s, 1)
        assert ctx.tree_info()[1] == 1
        res.append(s.numpy())
    for k in ("x", "vx", "ax_s", "ay_s", "az_s", "ax_h", "ay_h", "az_h"):
        a, b = (r[k][np.argsort(r["id"])] for r in res)
        if prec == 0:
            assert np.array_equal(a, b), k
        else:
            assert np.max(np.abs(a - b)) <= 1e-5 * np.max(np.abs(a)), k
