"""Tensor-core Gram and expansion where their tiles and loads end: rows around the 32-row
sub-chunks, the 256-row windows and the last of several parts; columns around the 8-, 64-
and 128-wide blocks; blocks with any row stride whose base is only element-aligned (scalar
loads) beside 16-byte aligned ones.

Tolerance: the claimed error of a window (expansion: of a row and column) is 2^-53
(float32 blocks: 2^-33) of rows x max|x| max|y|, and the reference is rounded by less than
2^-51 of sum |x||y| plus, for float32 results, 2^-24 of the value; 2^-50, 2^-31 and 2^-23
are allowed."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu

NS = [1, 31, 32, 33, 63, 65, 127, 129, 255, 256, 257, 511, 513, 39000]
KS = [1, 7, 8, 9, 33, 63, 64, 65, 127, 128]


def block(X, dtype, ld, off):
    """X in an [n][ld] block that starts `off` elements past a 256-byte boundary."""
    n, k = X.shape
    flat = torch.zeros(n * ld + off, dtype=dtype, device="cuda")
    T = flat[off:].view(n, ld)
    T[:, :k] = torch.from_numpy(X).to(dtype).cuda()
    return T


def layouts(dtype, k):
    a = 2 if dtype == torch.float64 else 4
    up = (k + a - 1) // a * a
    # float32 blocks keep ld % 4 == 0; any ld and any element alignment else
    return [(up, 0), (up + 2 * a, 1), (up + a + (1 if dtype == torch.float64 else 0), 0)]


@pytest.mark.parametrize("dtype", [torch.float64, torch.float32])
@pytest.mark.parametrize("k", KS)
def test_gram_edges(gpu_bmg, dtype, k):
    rng = np.random.default_rng(k)
    f64 = dtype == torch.float64
    for n in NS:
        X, Y = rng.standard_normal((n, k)), rng.standard_normal((n, k))
        if not f64:
            X, Y = X.astype(np.float32).astype(np.float64), Y.astype(np.float32).astype(np.float64)
        bound = np.zeros((k, k))
        for r0 in range(0, n, 256):
            xs, ys = np.abs(X[r0:r0 + 256]), np.abs(Y[r0:r0 + 256])
            bound += xs.shape[0] * np.outer(xs.max(axis=0), ys.max(axis=0))
        tol = (2.0 ** -50 if f64 else 2.0 ** -31) * bound + 2.0 ** -51 * (np.abs(X).T @ np.abs(Y))
        ref = X.T @ Y
        for ld, off in layouts(dtype, k):
            G = torch.full((k, k), np.nan, dtype=torch.float64, device="cuda")
            (gpu_bmg.gram_tc if f64 else gpu_bmg.gram_tc_f32)(block(X, dtype, ld, off), block(Y, dtype, ld, off), k, G)
            err = np.abs(G.cpu().numpy() - ref)
            assert np.all(err <= tol), (n, ld, off, (err / tol).max())


@pytest.mark.parametrize("dtype", [torch.float64, torch.float32])
@pytest.mark.parametrize("k", KS)
def test_expand_edges(gpu_bmg, dtype, k):
    rng = np.random.default_rng(100 + k)
    f64 = dtype == torch.float64
    for n in NS:
        X, Z, Yx = rng.standard_normal((n, k)), rng.standard_normal((n, k)), rng.standard_normal((k, k))
        if not f64:
            X, Z = X.astype(np.float32).astype(np.float64), Z.astype(np.float32).astype(np.float64)
        scale = np.abs(Z) + np.abs(X) @ np.abs(Yx)
        bound = k * np.outer(np.abs(X).max(axis=1), np.abs(Yx).max(axis=0))
        tol = 2.0 ** -50 * bound + 2.0 ** -51 * scale if f64 else 2.0 ** -31 * bound + 2.0 ** -23 * scale
        ref = Z + X @ Yx
        for ld, off in layouts(dtype, k):
            if ld % 2:
                continue                       # an expansion takes even strides
            U = block(np.full((n, ld), 7.0), dtype, ld, off)
            gpu_bmg.expand(block(Z, dtype, ld, off), block(X, dtype, ld, off), torch.from_numpy(Yx).cuda(), k, U, True)
            err = np.abs(U[:, :k].cpu().numpy().astype(np.float64) - ref)
            assert np.all(err <= tol), (n, ld, off, (err / tol).max())
            # columns from k on are written up to the end of the last 64-column block
            assert torch.all(U[:, k:(k + 63) // 64 * 64] == 0)
