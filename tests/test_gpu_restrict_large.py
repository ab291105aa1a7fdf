"""A restriction with more 16-byte chunks than one launch numbers: 162 rows of 13 300 000 float64
chunks, 2^31 < 162 * 13.3e6 (the prolongation's counterpart is in test_gpu_step_edges.py)."""
import pytest
import torch

from paper_1511_07042_gb300 import inputs

pytestmark = pytest.mark.gpu


def test_restrict_beyond_2_31_chunks(gpu_bmg):
    """Exact: small integers, halved once."""
    torch.cuda.empty_cache()
    free, _ = torch.cuda.mem_get_info()
    if free < 210 << 30:
        pytest.skip("needs 210 GB of device memory")
    v, t = inputs.icosahedron()
    p = gpu_bmg.Problem(v, t, 3)
    p.hierarchy(3)
    n, nc, ld = 642, 162, 26_600_000
    par = torch.from_numpy(p.mesh(3)[2].astype("int64"))
    row = torch.arange(n, dtype=torch.float64)
    want = torch.zeros(nc, dtype=torch.float64)
    for q in range(2):
        want.index_add_(0, par[:, q], 0.5 * row)
    R = torch.empty((n, ld), dtype=torch.float64, device="cuda")
    for i in range(n):
        R[i].fill_(float(i))
    R[:, -2:] = 0.0
    Z = torch.empty((nc, ld), dtype=torch.float64, device="cuda")
    Z.fill_(-1.0)
    p.restrict(3, R, Z, ld)
    del R
    for i in range(nc):
        low, high = torch.aminmax(Z[i, :-2])
        assert low.item() == high.item() == want[i].item(), i
        assert bool((Z[i, -2:] == 0.0).all()), i
    del Z
    torch.cuda.empty_cache()
    p.close()
