"""Exchanges of the eigensolve's cluster kernels where CTAs run out of rows before others: the
factorisation and the tridiagonalisation deal the rows to 8 CTAs, so that from 2 to 25 rows
the last steps reach CTAs without a row, with one row, and with one that leaves."""
import numpy as np
import pytest
import torch

from oracle import bmg as obmg

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", list(range(2, 18)) + [23, 24, 25])
@pytest.mark.parametrize("drop", [0, 1])
def test_few_rows(gpu_bmg, n, drop):
    """The values agree with the oracle's to 1e-10 of the largest (rounding of n 2^-53 |T| is
    far below), and repeated calls give the same bits."""
    rng = np.random.default_rng(100 * n + drop)
    r = n - drop                               # the last column repeats the first one
    S, B = rng.standard_normal((r, r)), rng.standard_normal((r, r))
    C = np.concatenate([np.eye(r), np.eye(r)[:, :drop]], axis=1)
    Ah, Mh = C.T @ (S + S.T) @ C, C.T @ (B @ B.T + r * np.eye(r)) @ C
    Ad, Md = torch.from_numpy(Ah).cuda(), torch.from_numpy(Mh).cuda()
    first = None
    for _ in range(10):
        th = torch.empty(r, dtype=torch.float64, device="cuda")
        Y = torch.empty((n, r), dtype=torch.float64, device="cuda")
        rk = torch.zeros(1, dtype=torch.int32, device="cuda")
        gpu_bmg.dense_eig(Ad, Md, 0.0, r, th, Y, rk)
        assert int(rk.item()) == r
        if first is None:
            first = th, Y
        assert torch.equal(th, first[0]) and torch.equal(Y, first[1])
    ref, _ = obmg.svqb_eig(Ah, Mh, 0.0, r)
    got, Yh = first[0].cpu().numpy(), first[1].cpu().numpy()
    assert np.allclose(got, ref, rtol=1e-10, atol=1e-10 * np.abs(ref).max())
    assert np.allclose(Yh.T @ Mh @ Yh, np.eye(r), atol=1e-11)
