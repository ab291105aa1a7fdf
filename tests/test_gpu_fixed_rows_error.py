"""Error of the float64 row products formed in integers on rows made for a large one: one product
that the dispatch just accepts (its factors near the smallest mantissas), the other values of X
2^-8 to 2^-12 as large with the low bits of their mantissas set, with the signs of the low
parts of the matrix values, so that what the integer sum drops adds up.

An integer sum has to be no worse than the float64 sum that it takes the place of: over all such
rows, neither its mean nor its largest error (over sum |a||x|) exceeds those of the chain of
float64 multiply-adds over the same rows, both against exact sums."""
import ctypes
import ctypes.util
from fractions import Fraction

import numpy as np
import pytest
import torch

from paper_1511_07042_gb300 import inputs

pytestmark = pytest.mark.gpu

fma = ctypes.CDLL(ctypes.util.find_library("m")).fma
fma.restype, fma.argtypes = ctypes.c_double, [ctypes.c_double] * 3


def low_sign(a, emax, bits):
    """Sign of the low part of a over 2^bits units, at 59 bits below 2^emax."""
    v = int(abs(Fraction(a)) * 2 ** 59 / Fraction(2) ** int(emax))
    low = (v + (1 << (bits - 1))) % (1 << bits) - (1 << (bits - 1))
    return (1 if low >= 0 else -1) * (1 if a >= 0 else -1)


@pytest.mark.parametrize("bits", [32, 29])   # a left-out half, and the present part
@pytest.mark.parametrize("which", [0, 1])
def test_error_no_larger_than_a_float64_sum(gpu_bmg, bits, which):
    v, t = inputs.icosahedron()
    p = gpu_bmg.Problem(v, t, 4, 0.1, inputs.sh_coefficients(3))
    p.hierarchy(2)
    rp, col, *vals = p.csr(4)
    val = vals[which]
    n, k, rng = rp.size - 1, 256, np.random.default_rng(bits + which)
    # rows of seven nonzeros whose diagonal is not among the first two
    rows = [i for i in range(n) if rp[i + 1] - rp[i] == 7 and list(col[rp[i]:rp[i + 1]]).index(i) >= 2]
    rows = rng.choice(rows, k)
    X = np.zeros((n, k))
    for c, i in enumerate(rows):
        b, d = rp[i], list(col[rp[i]:rp[i + 1]]).index(i)
        a = val[b:b + 7]
        emax = max(np.frexp(a[2:])[1])
        big = rng.choice([q for q in range(2, 7) if q != d])
        for q in range(2, 7):
            m = rng.integers(2 ** 52, 2 ** 52 + 2 ** 50)
            if q != big:               # the low bits of the half or part that is left out, all set
                m = (m >> (bits + 1) << (bits + 1)) | (2 ** bits - 2)
            x = float(m) * 2.0 ** -52 * (1.0 if q == big else 2.0 ** -int(rng.integers(8, 13)))
            X[col[b + q], c] = x * (1.0 if q == big else low_sign(a[q], emax, bits))
    Xd = torch.from_numpy(X).cuda()
    out = [torch.empty_like(Xd) for _ in range(2)]
    p.spmm(2, 2, Xd, k, *out)
    got = out[which].cpu().numpy()
    err, ref = [], []
    for c, i in enumerate(rows):
        a, x = val[rp[i]:rp[i + 1]], X[col[rp[i]:rp[i + 1]], c]
        exact = sum(Fraction(float(u)) * Fraction(float(w)) for u, w in zip(a, x))
        mag = sum(abs(Fraction(float(u)) * Fraction(float(w))) for u, w in zip(a, x))
        s = 0.0
        for u, w in zip(a, x):
            s = fma(float(u), float(w), s)
        err.append(float(abs(Fraction(float(got[i, c])) - exact) / mag))
        ref.append(float(abs(Fraction(s) - exact) / mag))
    print("integers: mean %.1e max %.1e, float64: mean %.1e max %.1e" % (np.mean(err), max(err), np.mean(ref), max(ref)))
    assert np.mean(err) <= np.mean(ref) and max(err) <= max(ref)
    p.close()
