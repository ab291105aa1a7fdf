"""Edges of the step kernels: the eigensolve at the sizes where its rows per warp and CTAs
change, with equal pivots and with dependent columns; Jacobi sweeps that alternate between
two blocks; row orders and colour groups of a level that the device sort takes in many
tiles; a prolongation with more chunks than one launch numbers."""
import numpy as np
import pytest
import scipy.sparse as sp
import torch

from oracle import bmg as obmg, multilevel
from paper_1511_07042_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def level6(gpu_bmg):
    """40962 rows: 21 tiles of the sort."""
    v, t = inputs.icosahedron()
    p = gpu_bmg.Problem(v, t, 6)
    p.hierarchy(3)
    rp, col, a, m = p.csr(6)
    n = rp.size - 1
    yield p, sp.csr_matrix((a, col, rp), (n, n)), sp.csr_matrix((m, col, rp), (n, n))
    p.close()


def dev(X, dtype=torch.float64):
    T = torch.zeros((X.shape[0], (X.shape[1] + 3) // 4 * 4), dtype=dtype, device="cuda")
    T[:, :X.shape[1]] = torch.from_numpy(X).to(dtype).cuda()
    return T


@pytest.mark.parametrize("n", [1, 2, 3, 8, 31, 32, 33, 63, 64, 65, 127, 129, 191, 193, 223, 224])
@pytest.mark.parametrize("kind", ["identity", "dependent"])
def test_dense_eig_sizes(gpu_bmg, n, kind):
    """identity: every pivot of the scaled matrix is 1 until the end.  dependent: the last
    columns repeat the first ones, so their pivots fall to rounding and are dropped.  The
    values agree with the oracle's to 1e-10 of the largest, as for other matrices of this
    size (rounding of n 2^-53 |T| is below 1e-13)."""
    rng = np.random.default_rng(n)
    S = rng.standard_normal((n, n))
    S = S + S.T
    r = n
    if kind == "identity":
        Mh, Ah = np.eye(n) * 2.0, S
    else:
        r = n - n // 4
        B = rng.standard_normal((r, r))
        C = np.concatenate([np.eye(r), np.eye(r)[:, :n - r]], axis=1)
        Mh, Ah = C.T @ (B @ B.T + r * np.eye(r)) @ C, C.T @ S[:r, :r] @ C
    k = max(1, r // 2)
    th = torch.empty(k, dtype=torch.float64, device="cuda")
    Y = torch.empty((n, k), dtype=torch.float64, device="cuda")
    rk = torch.zeros(1, dtype=torch.int32, device="cuda")
    gpu_bmg.dense_eig(torch.from_numpy(Ah).cuda(), torch.from_numpy(Mh).cuda(), 0.0, k, th, Y, rk)
    assert int(rk.item()) == r
    ref, _ = obmg.svqb_eig(Ah, Mh, 0.0, k)
    got, Yh = th.cpu().numpy(), Y.cpu().numpy()
    assert np.allclose(got, ref, rtol=1e-10, atol=1e-10 * np.abs(ref).max())
    assert np.allclose(Yh.T @ Mh @ Yh, np.eye(k), atol=1e-11)


@pytest.mark.parametrize("dtype", [torch.float64, torch.float32])
@pytest.mark.parametrize("nu", [1, 2, 3, 4, 5])
@pytest.mark.parametrize("with_b", [True, False])
def test_jacobi_sweeps_equal_single_sweeps(level6, dtype, nu, with_b):
    """nu sweeps of one call and nu calls of one sweep give the same bits."""
    p, A, M = level6
    rng = np.random.default_rng(nu)
    k, n = 12, A.shape[0]
    X, B = dev(rng.standard_normal((n, k)), dtype), dev(rng.standard_normal((n, k)), dtype)
    s = torch.from_numpy(rng.uniform(0, 9, k)).to(dtype).cuda()
    fn = p.smooth if dtype == torch.float64 else p.smooth_f32
    many, one, work = X.clone(), X.clone(), torch.empty_like(X)
    fn(3, 3, many, B if with_b else None, s, k, "jacobi", nu, 2 / 3, work)
    for _ in range(nu):
        fn(3, 3, one, B if with_b else None, s, k, "jacobi", 1, 2 / 3, work)
    assert torch.equal(many, one)


def test_row_order_and_colour_groups_of_a_large_level(level6):
    """Every row is visited once: A X and M X of a block that was NaN, and a symmetric
    Gauss-Seidel and a Kaczmarz sweep against the oracle's on the level's own colouring."""
    p, A, M = level6
    rng = np.random.default_rng(1)
    k, n = 4, A.shape[0]
    X, B, s = rng.standard_normal((n, k)), rng.standard_normal((n, k)), rng.uniform(0, 9, k)
    Xd, Bd = dev(X), dev(B)
    AX, MX = torch.full_like(Xd, np.nan), torch.full_like(Xd, np.nan)
    p.spmm(3, 3, Xd, k, AX, MX)
    # 12 products of float64 at most
    assert np.all(np.abs(AX.cpu().numpy() - A @ X) <= 2.0 ** -49 * (abs(A) @ np.abs(X)))
    assert np.all(np.abs(MX.cpu().numpy() - M @ X) <= 2.0 ** -49 * (abs(M) @ np.abs(X)))
    sd = torch.from_numpy(s).cuda()
    for smoother, ref in (("mcsgs", multilevel.mc_gauss_seidel(A, M, X, B, s, p.colouring(3)[0], 1, symmetric=True)),
                          ("kaczmarz", multilevel.kaczmarz(A, M, X, B, s, p.colouring2(3)[0], 1, 1.0))):
        Y = Xd.clone()
        p.smooth(3, 3, Y, Bd, sd, k, smoother, 1, 1.0, torch.empty_like(Xd))
        assert np.max(np.abs(Y.cpu().numpy() - ref)) <= 1e-12 * np.max(np.abs(ref)), smoother


def test_prolong_beyond_2_31_chunks(gpu_bmg):
    """642 rows of 3 400 000 float64 chunks (35 GB): 2^31 < 642 * 3.4e6.  Exact."""
    free, _ = torch.cuda.mem_get_info()
    if free < 80 << 30:
        pytest.skip("needs 80 GB of device memory")
    v, t = inputs.icosahedron()
    p = gpu_bmg.Problem(v, t, 3)
    p.hierarchy(3)
    n, nc, ld = 642, 162, 6_800_000
    par = torch.from_numpy(p.mesh(3)[2].astype(np.int64)).cuda()
    Xc = torch.empty((nc, ld), dtype=torch.float64, device="cuda")
    Xc.copy_(torch.arange(nc, dtype=torch.float64, device="cuda")[:, None])
    Xc[:, -2:] = 7.0
    Y = torch.full((n, ld), np.nan, dtype=torch.float64, device="cuda")
    p.prolong(3, Xc, Y, ld)
    want = (par[:, 0] + par[:, 1]).to(torch.float64) / 2
    for i in range(n):
        assert bool((Y[i, :-2] == want[i]).all()) and bool((Y[i, -2:] == 7.0).all()), i
    p.close()
