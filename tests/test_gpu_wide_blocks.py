"""Row kernels on blocks of more than 128 16-byte chunks (256 float64 or 512 float32 columns): the
same bits as on narrower blocks of the same columns."""
import numpy as np
import pytest
import torch

from paper_1511_07042_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dtype,k", [(torch.float64, 256), (torch.float64, 258), (torch.float64, 700),
                                     (torch.float32, 512), (torch.float32, 516), (torch.float32, 1300)])
def test_columns_beyond_a_slab(gpu_bmg, dtype, k):
    v, t = inputs.icosahedron()
    p = gpu_bmg.Problem(v, t, 3)
    p.hierarchy(2)
    n = inputs.n_vertices(3)
    f64 = dtype == torch.float64
    g = torch.Generator(device="cuda").manual_seed(k)
    X, B = (torch.randn((n, k), dtype=dtype, device="cuda", generator=g) for _ in range(2))
    s = torch.rand(k, dtype=dtype, device="cuda", generator=g)
    spmm, smooth = (p.spmm, p.smooth) if f64 else (p.spmm_f32, p.smooth_f32)

    def results(X, B, s):
        k = X.shape[1]
        out = [torch.full_like(X, np.nan) for _ in range(2)]
        spmm(2, 2, X, k, *out)
        for smoother in ("jacobi", "mcgs", "mcsgs", "kaczmarz"):
            out.append(X.clone())
            smooth(2, 2, out[-1], B, s, k, smoother, 2, 0.75 if smoother == "jacobi" else 1.0, torch.empty_like(X))
        return out

    parts = [results(X[:, c:c + 64].contiguous(), B[:, c:c + 64].contiguous(), s[c:c + 64].contiguous())
             for c in range(0, k, 64)]
    for q, out in enumerate(results(X, B, s)):
        assert torch.equal(out, torch.cat([part[q] for part in parts], dim=1)), q
    p.close()
