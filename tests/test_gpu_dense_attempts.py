"""Repeated attempts of the eigensolve: every attempt alone, pencils on which the first one does
not converge, matrices with NaN, and the bounded waits of its cluster exchanges.

Tolerance: an accepted solve has an error estimate (the off-diagonal norm of W^T T W over the
largest value, plus ||I - W^T W||) of at most 1e-6, and both the values and Y^T M Y - I are
within that estimate; 2e-6 is allowed."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu

TIMEOUT, NONFINITE = 9, 6


def spectrum(kind, n, rng):
    if kind == "groups":              # groups of one size, each of one value and its neighbours
        m = int(rng.integers(2, 39))
        return np.repeat(rng.uniform(0, 1, (n + m - 1) // m), m)[:n] * (
            1 + rng.uniform(-1, 1, n) * 10.0 ** rng.uniform(-12, -4))
    if kind == "wide groups":
        m = int(rng.integers(20, 40))
        return np.repeat(rng.uniform(0, 1, (n + m - 1) // m), m)[:n] + rng.uniform(-1, 1, n) * 10.0 ** rng.uniform(-5, -3)
    if kind == "geometric":           # more than 40 pairs below 1e-3 of the largest
        return np.geomspace(1e-8, 1, n)
    if kind == "one group":
        return 1 + 1e-4 * rng.random(n)
    return 1.0 + np.arange(n)


def pencil(kind, n, seed):
    rng = np.random.default_rng(seed)
    lam = spectrum(kind, n, rng)
    Q, _ = np.linalg.qr(rng.standard_normal((n, n)))
    A = torch.from_numpy((Q * lam) @ Q.T).cuda()
    return 0.5 * (A + A.T), torch.eye(n, dtype=torch.float64, device="cuda"), np.sort(lam)


def outputs(n):
    return (torch.empty(n, dtype=torch.float64, device="cuda"), torch.empty((n, n), dtype=torch.float64, device="cuda"))


def check(th, Y, ref, tol):
    assert np.abs(np.sort(th.cpu().numpy()) - ref).max() <= tol * np.abs(ref).max()
    assert (Y.T @ Y - torch.eye(len(ref), dtype=torch.float64, device="cuda")).abs().max().item() <= tol


@pytest.mark.parametrize("n", [1, 2, 33, 60, 170, 224])
@pytest.mark.parametrize("start", [0, 1, 2, 3])
def test_every_attempt(gpu_bmg, n, start):
    A, M, ref = pencil("plain", n, n)
    th, Y = outputs(n)
    assert gpu_bmg.dense_eig_attempt(A, M, 0.0, n, th, Y, start) <= 1e-10
    check(th, Y, ref, 1e-10)


@pytest.mark.parametrize("kind,n,seed", [("groups", 60, 1500), ("groups", 60, 2781), ("groups", 60, 3686),
                                         ("wide groups", 60, 1494), ("wide groups", 60, 2781), ("geometric", 60, 0),
                                         ("geometric", 224, 0), ("one group", 60, 0), ("one group", 200, 0)])
def test_first_attempt_does_not_converge(gpu_bmg, kind, n, seed):
    A, M, ref = pencil(kind, n, seed)
    th, Y = outputs(n)
    gpu_bmg.dense_eig(A, M, 0.0, n, th, Y)
    check(th, Y, ref, 2e-6)


def test_nan_is_reported(gpu_bmg):
    A, M, _ = pencil("plain", 40, 0)
    A[3, 3] = float("nan")
    with pytest.raises(gpu_bmg.BmgError) as e:
        gpu_bmg.dense_eig(A, M, 0.0, 8, *outputs(40))
    assert e.value.code == NONFINITE


def test_expired_waits_are_reported(gpu_bmg):
    """A row that sends nothing, in the factorisation and in the tridiagonalisation; a normal
    solve afterwards is right."""
    assert gpu_bmg.dense_timeout_selftest() == TIMEOUT
    assert "bounded wait" in gpu_bmg.LIB.bmg_last_error().decode()
    A, M, ref = pencil("plain", 40, 1)
    th, Y = outputs(40)
    gpu_bmg.dense_eig(A, M, 0.0, 40, th, Y)
    check(th, Y, ref, 1e-10)
