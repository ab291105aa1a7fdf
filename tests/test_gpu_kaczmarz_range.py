"""Kaczmarz sweeps with shifts so large that the squared row norms ||(A - s M) row||^2 leave the
range of float32: 2^128 and more in float64 blocks, where a sweep still projects every row as
the oracle's does, and float32 overflow in float32 blocks, where such a row is left as it is.

Tolerance: a projection rounds as in the sweeps of ordinary shifts, 1e-11 of the largest."""
import numpy as np
import pytest
import scipy.sparse as sp
import torch

from oracle import multilevel
from paper_1511_07042_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def level(gpu_bmg):
    v, t = inputs.icosahedron()
    p = gpu_bmg.Problem(v, t, 4)
    p.hierarchy(2)
    rp, col, a, m = p.csr(4)
    n = rp.size - 1
    yield p, sp.csr_matrix((a, col, rp), (n, n)), sp.csr_matrix((m, col, rp), (n, n))
    p.close()


@pytest.mark.parametrize("k", [2, 6, 34])
def test_norms_above_2_128(level, k):
    p, A, M = level
    rng = np.random.default_rng(k)
    n = A.shape[0]
    s = 10.0 ** np.resize([3.0, 17.0, 20.0, 23.0, 30.0, 60.0], k)   # squared norms of 1e0 to 1e114
    X = rng.standard_normal((n, k))
    B = rng.standard_normal((n, k)) * s * np.abs(M).sum(axis=1).max()
    B[:, ::3] = 0.0
    ref = multilevel.kaczmarz(A, M, X, B, s, p.colouring2(2)[0], 2, 1.0)
    Xd, Bd, sd = (torch.from_numpy(x).cuda() for x in (X, B, s))
    p.smooth(2, 2, Xd, Bd, sd, k, "kaczmarz", 2, 1.0, torch.empty_like(Xd))
    assert np.all(np.abs(Xd.cpu().numpy() - ref) <= 1e-11 * np.abs(ref).max(axis=0))


def test_float32_overflow_leaves_the_rows(level):
    p, A, _ = level
    X = torch.randn((A.shape[0], 4), device="cuda")
    Y, s = X.clone(), torch.full((4,), 1e23, device="cuda")
    p.smooth_f32(2, 2, Y, None, s, 4, "kaczmarz", 1, 1.0, torch.empty_like(X))
    assert torch.equal(X, Y)
