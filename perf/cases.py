"""The work a user of the library has it do, as timed cases: set-up, whole solves and the
steps of the cycle on device blocks, each through the public binding (bmg.py).

Sizes are those of the repository's workloads (inputs.WORKLOADS, the batched workload and
the parity tests).  `exact` restates each case in plain numpy and torch in 64 bits.
"""
import math

import numpy as np
import torch

from paper_1511_07042_gb300 import bmg, inputs

N1 = 42                       # vertices of level 1 (the icosahedron refined once)
SURFACE = (0.1, 1003)         # amplitude and harmonic seed of the perturbed sphere


# ------------------------------------------------------------------ the cases ----
def listed():
    return [
        # set-up of one surface of the batched workload: mesh, matrices, hierarchy
        {"name": "setup_r7", "kind": "setup", "r": 7},
        # the smallest surface of the batched workload, solved on its own: latency
        {"name": "solve_r4_k32", "kind": "solve", "r": 4, "k": 32, "wanted": 24, "tol": 1e-8,
         "smoother": "jacobi", "nu": 2, "coef_seed": SURFACE[1]},
        # the largest configuration: 655362-vertex unit sphere, 100 eigenvalues, float64
        {"name": "solve_r8_k128", "kind": "solve_sphere", "r": 8, "k": 128, "wanted": 100, "tol": 1e-8,
         "intermediate": 8},
        # [AX | MX] of the largest block (float64, smooth iterates of late cycles)
        {"name": "spmm_f64_r8_k128", "kind": "spmm", "r": 8, "k": 128, "f32": False},
        # the same product on a small level with an odd block (float32, a start block)
        {"name": "spmm_f32_r5_k33", "kind": "spmm", "r": 5, "k": 33, "f32": True},
        # damped Jacobi, two sweeps: the precision form's smoothing on the largest level
        {"name": "jacobi_f32_r8_k128", "kind": "smooth", "r": 8, "k": 128, "f32": True, "smoother": "jacobi", "nu": 2},
        # symmetric multicolour Gauss-Seidel of the 40962-vertex workload
        {"name": "mcsgs_f64_r6_k64", "kind": "smooth", "r": 6, "k": 64, "f32": False, "smoother": "mcsgs", "nu": 1},
        # five Kaczmarz sweeps of the interior workload (163842 vertices, k = 48)
        {"name": "kaczmarz_f64_r7_k48", "kind": "smooth", "r": 7, "k": 48, "f32": False, "smoother": "kaczmarz",
         "nu": 5},
        # restriction of a residual and prolongation of a correction on the largest level
        {"name": "transfer_r8_k128", "kind": "transfer", "r": 8, "k": 128},
        # Rayleigh-Ritz Gram product of the largest block
        {"name": "gram_f64_r8_k128", "kind": "gram", "r": 8, "k": 128, "f32": False},
        # Ritz vectors Z + X Y of an odd float32 block
        {"name": "expand_f32_r7_k99", "kind": "expand", "r": 7, "k": 99, "f32": True},
        # the enriched eigensolve of the largest workload's size, 42 + 128
        {"name": "dense_eig_k128", "kind": "dense", "r": 5, "k": 128},
    ]


def draw(rng):
    def log_int(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    kind = rng.choice(["setup", "solve", "spmm", "spmm", "jacobi", "mcsgs", "kaczmarz", "transfer", "gram", "gram",
                       "expand", "expand", "dense"])
    r = rng.randint(3, 8)
    k = log_int(4, 128)
    f32 = rng.random() < 0.5
    if kind == "setup":
        return {"kind": "setup", "r": rng.randint(3, 8)}
    if kind == "solve":
        k = rng.randint(16, 64)
        return {"kind": "solve", "r": rng.randint(4, 6), "k": k, "wanted": max(8, 3 * k // 4), "tol": 1e-8,
                "smoother": rng.choice(["jacobi", "mcsgs"]), "nu": rng.choice([1, 2]),
                "coef_seed": SURFACE[1] + rng.randint(0, 4)}
    if kind == "spmm":
        return {"kind": "spmm", "r": r, "k": k, "f32": f32}
    if kind in ("jacobi", "mcsgs", "kaczmarz"):
        return {"kind": "smooth", "r": r if kind == "jacobi" else min(r, 7), "k": k, "f32": f32, "smoother": kind,
                "nu": rng.randint(1, 3)}
    if kind == "transfer":
        return {"kind": "transfer", "r": max(r, 4), "k": k}
    if kind == "dense":
        return {"kind": "dense", "r": rng.randint(4, 6), "k": rng.randint(16, 160)}
    return {"kind": kind, "r": r, "k": k, "f32": f32}


# ----------------------------------------------------------------- the inputs ----
def _surface(r, amplitude=0.0, coefs=None, levels=None):
    v, t = inputs.icosahedron()
    p = bmg.Problem(v, t, r, amplitude, coefs)
    p.hierarchy(levels or r)
    return p


def _gen(seed):
    return torch.Generator(device="cuda").manual_seed(int(seed))


def _dtype(case):
    return torch.float32 if case.get("f32") else torch.float64


def _block(values, k, dtype):
    """[n][k] values as a k-interleaved block: the columns up to a multiple of 2 (4) zero."""
    a = 4 if dtype == torch.float32 else 2
    out = torch.zeros((values.shape[0], (k + a - 1) // a * a), dtype=dtype, device="cuda")
    out[:, :k] = values.to(dtype)
    return out


def _gauss(n, k, g):
    """A start block: N(0, 1) test vectors."""
    return torch.randn((n, k), dtype=torch.float64, device="cuda", generator=g)


def _waves(n, k, g):
    """Smooth iterates: plane waves over points of the unit sphere, the amplitude of unit
    M-norm vectors, with the roughness that an unconverged iterate still has."""
    V = torch.from_numpy(_points(n)).cuda()
    W = 3.0 * torch.randn((3, k), dtype=torch.float64, device="cuda", generator=g)
    ph = 2 * math.pi * torch.rand(k, dtype=torch.float64, device="cuda", generator=g)
    return torch.cos(V @ W + ph) * 0.4 + 1e-3 * _gauss(n, k, g)


def _points(n):
    r = int(round(math.log((n - 2) / 10, 4)))
    return _mesh(r)[0]


def _smooth_data(case, seed):
    n, k, g = inputs.n_vertices(case["r"]), case["k"], _gen(seed)
    X = _waves(n, k, g)
    B = _waves(n, k, g) * (100.0 / n)
    s = 20.0 * torch.rand(k, dtype=torch.float64, device="cuda", generator=g)
    dt = _dtype(case)
    return _block(X, k, dt), _block(B, k, dt), _block(s[None, :], k, dt)[0]


def _spmm_data(case, seed):
    n, k, g = inputs.n_vertices(case["r"]), case["k"], _gen(seed)
    return _block(_gauss(n, k, g) if case["f32"] else _waves(n, k, g), k, _dtype(case))


def _transfer_data(case, seed):
    nf, nc, k, g = inputs.n_vertices(case["r"]), inputs.n_vertices(case["r"] - 1), case["k"], _gen(seed)
    return tuple(_block(_waves(n, k, g), k, torch.float64) for n in (nf, nf, nc))   # residual, iterate, correction


def _gram_data(case, seed):
    n, k, g = inputs.n_vertices(case["r"]), case["k"], _gen(seed)
    return tuple(_block(_waves(n, k, g), k, _dtype(case)) for _ in range(2))


def _expand_data(case, seed):
    n, k, g = inputs.n_vertices(case["r"]), case["k"], _gen(seed)
    Z, X = (_block(_waves(n, k, g), k, _dtype(case)) for _ in range(2))
    Y = torch.randn((k, k), dtype=torch.float64, device="cuda", generator=g) / math.sqrt(k)
    return Z, X, Y


def _dense_data(case, seed):
    """Enriched matrices of a Gaussian block after two averaging steps: the shape and the
    conditioning of a first cycle's Rayleigh-Ritz (Q^T A Q, Q^T A X, X^T A X and with M)."""
    r, k, g = case["r"], case["k"], _gen(seed)
    V, T, parents = _mesh(r)
    cols, a, m = _operators(r)
    X = _gauss(V.shape[0], k, g)
    for _ in range(2):
        X = X - (2.0 / 3.0) * _apply(cols, a, X) / _diagonal(cols, a)[:, None]
    Q = torch.eye(N1, dtype=torch.float64, device="cuda")
    for q in range(2, r + 1):
        par = torch.from_numpy(_mesh(q)[2]).cuda().long()
        Q = 0.5 * (Q[par[:, 0]] + Q[par[:, 1]])
    E = torch.cat([Q, X], 1)
    S = [E.T @ _apply(cols, v, E) for v in (a, m)]
    return tuple(0.5 * (G + G.T) for G in S)


def prepare(case, seed):
    kind = case["kind"]
    if kind == "setup":
        return {"case": case, "mesh": inputs.icosahedron(), "coefs": inputs.sh_coefficients(seed % (1 << 31))}
    if kind in ("solve", "solve_sphere"):
        coefs = inputs.sh_coefficients(case["coef_seed"]) if kind == "solve" else None
        p = _surface(case["r"], SURFACE[0] if kind == "solve" else 0.0, coefs)
        n2, n = inputs.n_vertices(2), inputs.n_vertices(case["r"])
        st = {"case": case, "p": p, "X0": _gauss(n2, case["k"], _gen(seed))}
        if kind == "solve":
            st["U"] = torch.empty((n, case["wanted"]), dtype=torch.float64, device="cuda")
            st["opt"] = bmg.options(smoother=case["smoother"], nu=case["nu"])
        else:
            st["opt"] = bmg.options(cycles_intermediate=case["intermediate"])
        return st
    if kind == "spmm":
        X = _spmm_data(case, seed)
        return {"case": case, "p": _surface(case["r"]), "X": X, "AX": torch.empty_like(X), "MX": torch.empty_like(X)}
    if kind == "smooth":
        X, B, s = _smooth_data(case, seed)
        return {"case": case, "p": _surface(case["r"]), "X": X, "B": B, "s": s, "work": torch.empty_like(X)}
    if kind == "transfer":
        R, Y, C = _transfer_data(case, seed)
        return {"case": case, "p": _surface(case["r"]), "R": R, "Y": Y, "C": C, "Z": torch.empty_like(C)}
    if kind == "gram":
        X, Y = _gram_data(case, seed)
        return {"case": case, "X": X, "Y": Y, "G": torch.empty((case["k"],) * 2, dtype=torch.float64, device="cuda")}
    if kind == "expand":
        Z, X, Y = _expand_data(case, seed)
        return {"case": case, "Z": Z, "X": X, "Y": Y, "U": torch.empty_like(X)}
    A, M = _dense_data(case, seed)
    k = case["k"]
    return {"case": case, "A": A, "M": M, "theta": torch.empty(k, dtype=torch.float64, device="cuda"),
            "Y": torch.empty((N1 + k, k), dtype=torch.float64, device="cuda")}


# -------------------------------------------------------------------- one pass ----
def run(st):
    case = st["case"]
    kind, r, k = case["kind"], case["r"], case.get("k")
    if kind == "setup":
        v, t = st["mesh"]
        p = bmg.Problem(v, t, r, SURFACE[0], st["coefs"])
        p.hierarchy(r)
        out = [p.mesh(r)[0]] + list(p.csr(r)) + [p.colouring(r)[0]]
        p.close()
        return out
    if kind == "solve":
        # the residual norms, formed by cancellation, are left to the solver's own test
        ev, U, _, _ = st["p"].solve(st["X0"], k, case["wanted"], 0.0, case["tol"], st["opt"], evecs_device=st["U"])
        return [ev, U]
    if kind == "solve_sphere":
        # eigenvalues only, as the option has it: the sphere's multiplets fix no vectors
        return [st["p"].solve(st["X0"], k, case["wanted"], 0.0, case["tol"], st["opt"], evecs=False)[0]]
    if kind == "spmm":
        (st["p"].spmm_f32 if case["f32"] else st["p"].spmm)(r, r, st["X"], k, st["AX"], st["MX"])
        return [st["AX"], st["MX"]]
    if kind == "smooth":
        fn = st["p"].smooth_f32 if case["f32"] else st["p"].smooth
        omega = 2.0 / 3.0 if case["smoother"] == "jacobi" else 1.0
        fn(r, r, st["X"], st["B"], st["s"], k, case["smoother"], case["nu"], omega, st["work"])
        return [st["X"]]
    if kind == "transfer":
        st["p"].restrict(r, st["R"], st["Z"], k)
        st["p"].prolong(r, st["C"], st["Y"], k, add=True)
        return [st["Z"], st["Y"]]
    if kind == "gram":
        (bmg.gram_tc_f32 if case["f32"] else bmg.gram_tc)(st["X"], st["Y"], k, st["G"])
        return [st["G"]]
    if kind == "expand":
        bmg.expand(st["Z"], st["X"], st["Y"], k, st["U"])
        return [st["U"]]
    bmg.dense_eig(st["A"], st["M"], 0.0, k, st["theta"], st["Y"])
    return [st["theta"], st["Y"]]


# ---------------------------------------------------------- what it has to do ----
def work(case):
    kind, r, k = case["kind"], case["r"], case.get("k", 0)
    T = 4.0 if case.get("f32") else 8.0
    n = float(inputs.n_vertices(r))
    nnz = 7.0 * n - 12.0
    nc = (n + 6.0) / 4.0
    csr = (4.0 + 2.0 * T) * nnz + 4.0 * n
    if kind == "setup":   # vertices, pattern and values of every refinement written once
        return {"bytes": 4.0 / 3.0 * (24.0 * n + 24.0 * n + 20.0 * nnz + 4.0 * n), "flops": 4.0 / 3.0 * 100.0 * 2.0 * n}
    if kind in ("solve", "solve_sphere"):
        h = float(N1 + k)
        flops = 0.0
        for q in range(2, r + 1):   # 8 cycles a level: two products, two sweeps, two Grams, expansion, eigensolve
            m = float(inputs.n_vertices(q))
            flops += 8.0 * (8.0 * 7.0 * m * k + 3.0 * 2.0 * 7.0 * m * k + 3.0 * 2.0 * m * k * k + 9.0 * h ** 3)
        return {"bytes": csr + 8.0 * 162.0 * k + (8.0 * n * case["wanted"] if kind == "solve" else 0.0), "flops": flops}
    if kind == "spmm":
        return {"bytes": csr + 3.0 * T * n * k, "flops": 4.0 * nnz * k}
    if kind == "smooth":
        sweeps = case["nu"] * (2 if case["smoother"] == "mcsgs" else 1)
        per = (8.0 if case["smoother"] == "kaczmarz" else 4.0) * nnz * k + 6.0 * n * k
        return {"bytes": csr + 2.0 * T * n + 3.0 * T * n * k, "flops": sweeps * per}
    if kind == "transfer":
        return {"bytes": 8.0 * n + 8.0 * 7.0 * nc + T * k * (3.0 * n + 2.0 * nc), "flops": 4.0 * n * k}
    if kind == "gram":
        return {"bytes": 2.0 * T * n * k + 8.0 * k * k, "flops": 2.0 * n * k * k}
    if kind == "expand":
        return {"bytes": 3.0 * T * n * k + 8.0 * k * k, "flops": 2.0 * n * k * k}
    h = float(N1 + k)
    return {"bytes": 16.0 * h * h + 8.0 * h * k, "flops": 9.0 * h ** 3}


# ------------------------------------------- the same in plain numpy and torch ----
def _harmonics(n):
    """Real orthonormal spherical harmonics l <= 4 at unit vectors, l = 0..4, m = -l..l."""
    x, y, z = n[:, 0], n[:, 1], n[:, 2]
    c, s = [np.ones_like(x)], [np.zeros_like(x)]    # (sin theta)^m cos / sin (m phi)
    for m in range(4):
        c.append(x * c[m] - y * s[m])
        s.append(x * s[m] + y * c[m])
    P = {}
    for m in range(5):                              # Legendre functions over (sin theta)^m
        P[m, m] = np.full_like(x, float(np.prod(np.arange(1, 2 * m, 2))))
        for l in range(m + 1, 5):
            P[l, m] = ((2 * l - 1) * z * P[l - 1, m] - (l + m - 1) * P.get((l - 2, m), 0.0)) / (l - m)
    out = []
    for l in range(5):
        for m in range(-l, l + 1):
            a = abs(m)
            N = math.sqrt((2 * l + 1) / (4 * math.pi) * math.factorial(l - a) / math.factorial(l + a))
            out.append(N * P[l, a] * (1.0 if m == 0 else math.sqrt(2.0) * (c[a] if m > 0 else s[a])))
    return np.stack(out, 1)


def _project(m, amplitude, coefs):
    n = m / np.linalg.norm(m, axis=1)[:, None]
    return n if amplitude == 0.0 else (1.0 + amplitude * (_harmonics(n) @ coefs))[:, None] * n


_meshes = {}


def _mesh(r, amplitude=0.0, coefs=None):
    """Vertices, triangles and parents of the icosahedron refined r times (unit sphere: kept)."""
    if amplitude == 0.0 and r in _meshes:
        return _meshes[r]
    if r == 0:
        v, t = inputs.icosahedron()
        out = _project(v, amplitude, coefs), t.astype(np.int64), np.stack([np.arange(12)] * 2, 1)
    else:
        v, t, _ = _mesh(r - 1, amplitude, coefs)
        n = v.shape[0]
        ends = np.sort(t[:, [[0, 1], [1, 2], [2, 0]]], axis=2)
        key, at = np.unique(ends[..., 0] * n + ends[..., 1], return_inverse=True)
        e = np.stack([key // n, key % n], 1)
        new = _project(0.5 * (v[e[:, 0]] + v[e[:, 1]]), amplitude, coefs)
        ab, bc, ca = (n + at.reshape(-1, 3)).T
        a, b, c = t.T
        child = np.stack([a, ab, ca, b, bc, ab, c, ca, bc, ab, bc, ca], 1).reshape(-1, 3)
        out = np.concatenate([v, new]), child, np.concatenate([np.stack([np.arange(n)] * 2, 1), e])
    if amplitude == 0.0:
        _meshes[r] = out
    return out


def _csr(v, t):
    """P1 stiffness and mass on flat triangles: row starts, columns, values."""
    n = v.shape[0]
    p = [v[t[:, q]] for q in range(3)]
    cot, area = [], None
    for q in range(3):
        u, w = p[(q + 1) % 3] - p[q], p[(q + 2) % 3] - p[q]
        x = np.linalg.norm(np.cross(u, w), axis=1)
        cot.append((u * w).sum(1) / x)
        area = 0.5 * x if area is None else area
    i, j, a, m = [], [], [], []
    for q in range(3):
        s, w = (q + 1) % 3, (q + 2) % 3
        i += [t[:, q], t[:, s], t[:, w]]
        j += [t[:, q], t[:, w], t[:, s]]
        a += [0.5 * (cot[s] + cot[w]), -0.5 * cot[q], -0.5 * cot[q]]
        m += [area / 6.0, area / 12.0, area / 12.0]
    key, at = np.unique(np.concatenate(i) * n + np.concatenate(j), return_inverse=True)
    a, m = (np.bincount(at, np.concatenate(x), key.size) for x in (a, m))
    start = np.searchsorted(key, np.arange(n + 1) * n)
    return start, key % n, a, m


def _operators(r):
    """Columns and values of A and M with the rows padded to one width, on the GPU."""
    v, t, _ = _mesh(r)
    start, col, a, m = _csr(v, t)
    n, wide = v.shape[0], int(np.diff(start).max())
    at = start[:-1, None] + np.arange(wide)
    ok = at < start[1:, None]
    at = np.minimum(at, col.size - 1)
    cols = np.where(ok, col[at], np.arange(n)[:, None])
    return tuple(torch.from_numpy(x).cuda() for x in (cols, np.where(ok, a[at], 0.0), np.where(ok, m[at], 0.0)))


def _apply(cols, val, X):
    out = torch.zeros((cols.shape[0], X.shape[1]), dtype=X.dtype, device=X.device)
    for q in range(cols.shape[1]):
        out += val[:, q, None] * X[cols[:, q]]
    return out


def _diagonal(cols, val):
    return (val * (cols == torch.arange(cols.shape[0], device=cols.device)[:, None])).sum(1)


def _colours(cols, distance):
    """Sequential greedy colours in descending (splitmix64(v), v) order."""
    nb = [set(x) for x in cols.cpu().tolist()]
    n = len(nb)
    v = np.arange(n, dtype=np.uint64)
    with np.errstate(over="ignore"):
        z = v + np.uint64(0x9E3779B97F4A7C15)
        z = (z ^ (z >> np.uint64(30))) * np.uint64(0xBF58476D1CE4E5B9)
        z = (z ^ (z >> np.uint64(27))) * np.uint64(0x94D049BB133111EB)
        z = z ^ (z >> np.uint64(31))
    colour = [-1] * n
    for i in np.lexsort((v, z))[::-1].tolist():
        near = nb[i] if distance == 1 else set().union(*(nb[j] for j in nb[i]))
        used = {colour[j] for j in near}
        c = 0
        while c in used:
            c += 1
        colour[i] = c
    return torch.tensor(colour, device="cuda")


def _exact_smooth(case, seed):
    X, B, s = (x.double() for x in _smooth_data(case, seed))
    cols, a, m = _operators(case["r"])
    if case["f32"]:      # the precision form's operators are float32 copies
        a, m = a.float().double(), m.float().double()
    da, dm = _diagonal(cols, a), _diagonal(cols, m)
    if case["smoother"] == "jacobi":
        for _ in range(case["nu"]):
            res = B - _apply(cols, a, X) + s * _apply(cols, m, X)
            X = X + (2.0 / 3.0) * res / (da[:, None] - s * dm[:, None])
        return [X]
    colour = _colours(cols, 1 if case["smoother"] == "mcsgs" else 2)
    rows = [torch.nonzero(colour == c)[:, 0] for c in range(int(colour.max()) + 1)]
    order = rows + rows[::-1] if case["smoother"] == "mcsgs" else rows
    for _ in range(case["nu"]):
        for i in order:
            res = B[i] - _apply(cols[i], a[i], X) + s * _apply(cols[i], m[i], X)
            if case["smoother"] == "mcsgs":
                X[i] += res / (da[i, None] - s * dm[i, None])
                continue
            norm = sum((a[i, q, None] - s * m[i, q, None]) ** 2 for q in range(cols.shape[1]))
            for q in range(cols.shape[1]):
                X.index_add_(0, cols[i, q], res / norm * (a[i, q, None] - s * m[i, q, None]))
    return [X]


def exact(case, seed):
    kind, r, k = case["kind"], case["r"], case.get("k")
    if kind == "setup":
        v, t, _ = _mesh(r, SURFACE[0], inputs.sh_coefficients(seed % (1 << 31)))
        _, _, a, m = _csr(v, t)
        return [v, None, None, a, m, None]
    if kind == "solve_sphere":
        return None          # no closed form on the discrete surface; a dense solve is out of reach
    if kind == "solve":
        if r > 4:
            return None
        start, col, a, m = _csr(*_mesh(r, SURFACE[0], inputs.sh_coefficients(case["coef_seed"]))[:2])
        n = start.size - 1
        A, M = (np.zeros((n, n)) for _ in range(2))
        i = np.repeat(np.arange(n), np.diff(start))
        A[i, col], M[i, col] = a, m
        A, M = torch.from_numpy(A).cuda(), torch.from_numpy(M).cuda()
        L = torch.linalg.cholesky(M)
        S = torch.linalg.solve_triangular(L, torch.linalg.solve_triangular(L, A, upper=False).T, upper=False)
        return [torch.linalg.eigvalsh(0.5 * (S + S.T))[: case["wanted"]].cpu().numpy(), None]
    if kind == "spmm":
        X = _spmm_data(case, seed).double()
        cols, a, m = _operators(r)
        if case["f32"]:
            a, m = a.float().double(), m.float().double()
        return [_apply(cols, a, X), _apply(cols, m, X)]
    if kind == "smooth":
        return _exact_smooth(case, seed)
    if kind == "transfer":
        R, Y, C = _transfer_data(case, seed)
        par = torch.from_numpy(_mesh(r)[2]).cuda()
        Z = torch.zeros_like(C)
        for q in range(2):
            Z.index_add_(0, par[:, q], 0.5 * R)
        return [Z, Y + 0.5 * (C[par[:, 0]] + C[par[:, 1]])]
    if kind == "gram":
        X, Y = (b[:, :k].double() for b in _gram_data(case, seed))
        return [X.T @ Y]
    if kind == "expand":
        Z, X, Y = (b.double() for b in _expand_data(case, seed))
        U = Z.clone()
        U[:, :k] += X[:, :k] @ Y
        return [U]
    A, M = (x.cpu().numpy() for x in _dense_data(case, seed))
    L = np.linalg.cholesky(M)
    S = np.linalg.solve(L, np.linalg.solve(L, A).T)
    w = np.linalg.eigvalsh(0.5 * (S + S.T))
    return [w[np.argsort(np.abs(w), kind="stable")[:k]], None]
