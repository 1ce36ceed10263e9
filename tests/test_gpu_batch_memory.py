"""Device memory of batches of very many very small systems."""
import numpy as np
import pytest

from paper_1406_6158_gb300 import ics
from test_gpu_parity import H  # noqa: F401

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


def batch(H, S, n):
    """S systems of n particles, one after another in the same arrays."""
    st = ics.plummer(S * n, 3)
    t = {k: torch.as_tensor(st[k], device="cuda") for k in H.System.FIELDS}
    t.update({"a%s_%s" % (d, w): torch.zeros(S * n, device="cuda") for d in "xyz" for w in "sh"})
    arr = (H.hybrid_system * S)()
    for k, v in t.items():
        p, b = v.data_ptr(), v.element_size() * n
        for s in range(S):
            setattr(arr[s], k, p + s * b)
    for s in range(S):
        arr[s].n = n
    return t, arr


# A context's buffers per system: 16 KiB of radix counters (8 KiB for the system, 8 KiB for its one tile), and what its
# particles take. 1536 bytes each are what the server charges for a particle with its own 84 bytes of arrays; 1 KiB for
# the tables with one entry per system.
@pytest.mark.parametrize("n", [1, 8])
def test_memory_per_system(H, n):  # noqa: F811
    used = []
    for S in (20000, 80000):
        t, arr = batch(H, S, n)
        torch.cuda.synchronize()
        ctx = H.Context(H.Params(eps=0.05, theta=0.5, R1=0.1, R2=0.2))
        before = torch.cuda.mem_get_info()[0]
        assert ctx.L.hybrid_step_batched(ctx.h, arr, S, 1) == 0
        used.append(before - torch.cuda.mem_get_info()[0])
        assert np.isfinite(t["x"].cpu().numpy()).all()
        ctx.close()
    assert (used[1] - used[0]) / 60000 <= 16384 + 1024 + n * 1536
