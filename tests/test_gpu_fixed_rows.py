"""Float64 row products formed in integers (csrc/ops.cu, gather_row_fixed): values that take
the integer sum, values that must take the float64 loop (wide exponents, subnormals, Inf,
NaN, rows longer than seven nonzeros), and mixtures of both in one row.

Tolerance: a float64 sum of n products errs by at most n 2^-53 sum |a||x| and the integer
sum by less (its units are below 2^-53 of the row's largest product), so 2^-50 sum |a||x|
covers both sides for rows of up to 12 nonzeros; a result below 2^-1021 may lose its last
bits."""
import numpy as np
import pytest
import torch

from paper_1511_07042_gb300 import inputs

pytestmark = pytest.mark.gpu


def bipyramid(m):
    """Two poles over an m-gon: pole rows of m + 1 nonzeros after refinement."""
    a = 2 * np.pi * np.arange(m) / m
    v = np.concatenate([np.stack([np.cos(a), np.sin(a), 0 * a], 1), [[0, 0, 1.0], [0, 0, -1.0]]])
    t = [[i, (i + 1) % m, m] for i in range(m)] + [[(i + 1) % m, i, m + 1] for i in range(m)]
    return v, np.array(t, np.int32)


def values(kind, n, k, rng):
    X = rng.standard_normal((n, k))
    if kind == "wide":                # exponents that differ within a row
        X *= 2.0 ** rng.integers(-30, 31, (n, k))
    elif kind == "huge":              # outside the band of the integer sum, zeros between
        X *= 2.0 ** rng.choice([-1000, 0, 990], (1, k))
        X[rng.random((n, k)) < 0.3] = 0.0
    elif kind == "subnormal":
        X *= 2.0 ** rng.choice([-1070, -1040, 0], (n, k))
    elif kind == "local":             # zero but for one vertex a column, signed zeros
        keep = np.zeros((n, k), bool)
        keep[rng.integers(0, n, k), np.arange(k)] = True
        X = np.where(keep, X, -0.0)
    elif kind == "nonfinite":
        X[rng.integers(0, n, 40), rng.integers(0, k, 40)] = rng.choice([np.inf, -np.inf, np.nan], 40)
    return X


@pytest.mark.parametrize("mesh", ["ico", "bipyramid"])
@pytest.mark.parametrize("kind", ["normal", "wide", "huge", "subnormal", "local", "nonfinite"])
@pytest.mark.parametrize("k", [1, 7, 32, 66, 130])
def test_spmm_values(gpu_bmg, mesh, kind, k):
    v, t = inputs.icosahedron() if mesh == "ico" else bipyramid(11)
    p = gpu_bmg.Problem(v, t, 3)
    p.hierarchy(2)
    rp, col, a, m = p.csr(3)
    n = rp.size - 1
    X = values(kind, n, k, np.random.default_rng(17 + k))
    ld = (k + 1) // 2 * 2
    Xd = torch.zeros((n, ld), dtype=torch.float64, device="cuda")
    Xd[:, :k] = torch.from_numpy(X).cuda()
    AX, MX = torch.full_like(Xd, 3.0), torch.full_like(Xd, 3.0)
    p.spmm(2, 2, Xd, k, AX, MX)
    rows = np.repeat(np.arange(n), np.diff(rp))
    for out, val in ((AX, a), (MX, m)):
        got = out.cpu().numpy()
        assert np.all(got[:, k:] == 0)
        with np.errstate(invalid="ignore", over="ignore", under="ignore"):
            terms = val[:, None] * X[col]
            ref, mag = np.zeros((n, k)), np.zeros((n, k))
            np.add.at(ref, rows, terms)
            np.add.at(mag, rows, np.abs(terms))
        fine = np.isfinite(mag)
        assert np.array_equal(np.isnan(got[:, :k]), np.isnan(ref))
        assert np.array_equal(got[:, :k][~fine & ~np.isnan(ref)], ref[~fine & ~np.isnan(ref)])
        err = np.abs(got[:, :k][fine] - ref[fine])
        assert np.all(err <= 2.0 ** -50 * mag[fine] + 2.0 ** -1070), err.max()
        if kind == "local":           # rows that do not touch the vertex are exactly zero
            assert np.all(got[:, :k][mag == 0] == 0)
    p.close()
