"""Rows of more than seven nonzeros in the float64 row kernels (the first seven in integers and
the others one at a time, or the whole row one at a time): poles of 7 to 21 neighbours and a
mesh of random valences, at widths that give a row a part of a warp and a whole one.

Tolerance of the products: an integer sum of seven errs by less than 4 2^-53 sum |a||x|, each
further nonzero by one rounding, and the reference by one for each nonzero: (2 n + 4) 2^-53 for
rows of n."""
import numpy as np
import pytest
import scipy.sparse as sp
import torch
from scipy.spatial import ConvexHull

from oracle import multilevel

pytestmark = pytest.mark.gpu


def bipyramid(m):
    a = 2 * np.pi * np.arange(m) / m
    v = np.concatenate([np.stack([np.cos(a), np.sin(a), 0 * a], 1), [[0, 0, 1.0], [0, 0, -1.0]]])
    t = [[i, (i + 1) % m, m] for i in range(m)] + [[(i + 1) % m, i, m + 1] for i in range(m)]
    return v, np.array(t, np.int32)


def hull(n):
    v = np.random.default_rng(n).standard_normal((n, 3))
    v /= np.linalg.norm(v, axis=1)[:, None]
    t = ConvexHull(v).simplices.astype(np.int32)
    inward = np.einsum("ij,ij->i", np.cross(v[t[:, 1]] - v[t[:, 0]], v[t[:, 2]] - v[t[:, 0]]), v[t[:, 0]]) < 0
    t[inward] = t[inward][:, [0, 2, 1]]
    return v, t


@pytest.mark.parametrize("mesh", [7, 8, 9, 20, "hull"])
@pytest.mark.parametrize("k", [4, 20, 64, 130])
def test_long_rows(gpu_bmg, mesh, k):
    p = gpu_bmg.Problem(*(hull(300) if mesh == "hull" else bipyramid(mesh)), 3)
    p.hierarchy(2)
    rp, col, a, m = p.csr(3)
    n, rng = rp.size - 1, np.random.default_rng(k)
    assert np.diff(rp).max() > 7
    A, M = sp.csr_matrix((a, col, rp), (n, n)), sp.csr_matrix((m, col, rp), (n, n))
    X, B, s = rng.standard_normal((n, k)), rng.standard_normal((n, k)), rng.uniform(0, 0.5, k)
    Xd, Bd, sd = (torch.from_numpy(x).cuda() for x in (X, B, s))
    AX, MX = torch.full_like(Xd, np.nan), torch.full_like(Xd, np.nan)
    p.spmm(2, 2, Xd, k, AX, MX)
    tol = ((2 * np.diff(rp) + 4) * 2.0 ** -53)[:, None]
    assert np.all(np.abs(AX.cpu().numpy() - A @ X) <= tol * (abs(A) @ np.abs(X)))
    assert np.all(np.abs(MX.cpu().numpy() - M @ X) <= tol * (abs(M) @ np.abs(X)))
    for smoother, omega, ref in (
            ("jacobi", 2 / 3, X + 2 / 3 * (B - A @ X + s * (M @ X)) / (A.diagonal()[:, None] - s * M.diagonal()[:, None])),
            ("mcsgs", 1.0, multilevel.mc_gauss_seidel(A, M, X, B, s, p.colouring(2)[0], 1, symmetric=True)),
            ("kaczmarz", 1.0, multilevel.kaczmarz(A, M, X, B, s, p.colouring2(2)[0], 1, 1.0))):
        Y = Xd.clone()
        p.smooth(2, 2, Y, Bd, sd, k, smoother, 1, omega, torch.empty_like(Xd))
        assert np.max(np.abs(Y.cpu().numpy() - ref)) <= 1e-11 * np.max(np.abs(ref)), smoother
    p.close()
