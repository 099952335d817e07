"""Workloads that the performance of this library is measured on.

Each case is one call (or one step) that a user of the library makes, through
the public Python entry points, at sizes of this repository's benchmark,
configurations and tests: the sparse product S X, the Gram products and the
basis update in FP64 and in the mixed path's tensor-core form, the dense Ritz
solve, the shifted sparse solve, the shape gradient, a whole hierarchical solve
and a batch of them.  ``draw`` gives further cases of the same kinds over the
whole range: 4,096 to 10^6 rows, 20 to 500 eigenpairs (30 to 750 columns).

Meshes are bumpy tori (R = 1, r = 0.3) on an nu x nv grid with jitter and
Gaussian bumps, every draw and seed its own; bases are dense random blocks
scaled like M-orthonormal eigenvector blocks.
"""
import math

import numpy as np
import torch

import paper_2111_09039_gb300 as hs

DEV = "cuda:0"


# ---- the cases ------------------------------------------------------------------

def listed():
    return [
        # S X on the smallest mesh (64 x 64 torus, q = 30 columns of p = 20): a
        # call bound by launches and latency
        {"name": "spmm_small", "op": "spmm", "nu": 64, "nv": 64, "k": 30, "locked": 0},
        # S X of the benchmark's finest level, the whole subspace (q = 750)
        {"name": "spmm_large", "op": "spmm", "nu": 1000, "nv": 1000, "k": 750, "locked": 0},
        # reduced matrix Psi^T S Psi of the default (FP64) path: 163,842-vertex
        # sphere, p = 200 -> q = 300
        {"name": "gram_fp64", "op": "gram", "n": 163842, "k": 300, "tc": False, "digits": 0},
        # the same product as the mixed path takes it at tol 1e-5 (five digits),
        # 250,000 vertices, q = 750
        {"name": "gram_mixed", "op": "gram", "n": 250000, "k": 750, "tc": True, "digits": 5},
        # basis update Phi = Psi Phi_bar of the two paths at the same sizes
        {"name": "update_fp64", "op": "update", "n": 163842, "k": 300, "tc": False},
        {"name": "update_mixed", "op": "update", "n": 250000, "k": 750, "tc": True},
        # Ritz solve of a small problem (p = 50 -> q = 75), FP64 path
        {"name": "ritz_small", "op": "ritz", "k": 75, "tc": False},
        # Ritz solve of the benchmark (q = 750), mixed path, reduced mass near I
        # as after the first iteration of a level
        {"name": "ritz_large", "op": "ritz", "k": 750, "tc": True},
        # factorisation of S - mu M at a shift inside the spectrum and 75
        # right-hand sides (one inverse iteration of the FP64 path, p = 50)
        {"name": "shifted_solve", "op": "shifted_solve", "nu": 128, "nv": 128, "k": 75, "f32": False},
        # backward pass of the spectral loss: 40,000 vertices, 50 eigenpairs
        {"name": "eig_grad", "op": "eig_grad", "nu": 250, "nv": 160, "p": 50},
        # whole solve: 250,000-vertex torus, the benchmark's p = 500 and
        # tolerance, mixed precision, three levels
        {"name": "solve_mixed", "op": "solve", "nu": 500, "nv": 500, "p": 500, "levels": 3, "mixed": True, "tol": 1e-5},
        # a collection of 16 meshes of 5,000 to 80,000 vertices, 50 eigenpairs
        # each, solved concurrently
        {"name": "solve_batch", "op": "batch", "count": 16, "lo": 5000, "hi": 80000, "p": 50, "tol": 1e-5},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _grid(rng, lo, hi):
    """nu, nv of a torus of lo .. hi vertices, aspect 0.5 to 2 (odd sizes among them)."""
    n, a = _log(rng, lo, hi), rng.uniform(0.7, 1.4)
    nu = max(40, int(round(math.sqrt(n) * a)))
    return nu, max(40, int(round(n / nu)))


def draw(rng):
    op = rng.choice(["spmm", "spmm", "gram", "gram", "update", "update", "ritz", "ritz", "shifted_solve", "eig_grad",
                     "solve", "solve", "batch"])
    if op == "spmm":
        nu, nv = _grid(rng, 4096, 1000000)
        k = _log(rng, 30, 750)
        # the active columns of a block whose leading `locked` columns converged
        return {"op": op, "nu": nu, "nv": nv, "k": k, "locked": rng.choice([0, rng.randrange(0, k // 2)])}
    if op == "gram":
        tc = rng.random() < 0.5
        n, k = _log(rng, 4096, 250000), _log(rng, 30, 750 if tc else 300)
        return {"op": op, "n": n, "k": k, "tc": tc, "digits": rng.choice([5, 6]) if tc else 0}
    if op == "update":
        tc = rng.random() < 0.5
        return {"op": op, "n": _log(rng, 4096, 250000), "k": _log(rng, 30, 750 if tc else 300), "tc": tc}
    if op == "ritz":
        return {"op": op, "k": _log(rng, 30, 750), "tc": rng.random() < 0.5}
    if op == "shifted_solve":
        nu, nv = _grid(rng, 4096, 60000)
        return {"op": op, "nu": nu, "nv": nv, "k": _log(rng, 30, 300), "f32": rng.random() < 0.5}
    if op == "eig_grad":
        nu, nv = _grid(rng, 4096, 160000)
        return {"op": op, "nu": nu, "nv": nv, "p": _log(rng, 20, 100)}
    if op == "solve":
        mixed = rng.random() < 0.6
        nu, nv = _grid(rng, 5000, 160000 if mixed else 40000)
        return {"op": op, "nu": nu, "nv": nv, "p": _log(rng, 20, 300 if mixed else 100), "levels": rng.choice([2, 3]),
                "mixed": mixed, "tol": 1e-5 if mixed else 1e-8}
    return {"op": op, "count": rng.randrange(4, 13), "lo": 5000, "hi": _log(rng, 10000, 60000),
            "p": _log(rng, 20, 60), "tol": 1e-5}


# ---- inputs ---------------------------------------------------------------------

def _torus(nu, nv, seed):
    """Positions (n x 3) and triangles of a bumpy torus, vertex (i, j) at j * nu + i."""
    rng = np.random.default_rng(seed)
    n, du, dv = nu * nv, 2 * np.pi / nu, 2 * np.pi / nv
    i, j = np.tile(np.arange(nu), nv), np.repeat(np.arange(nv), nu)
    rad, ang = 0.1 * min(du, dv) * np.sqrt(rng.random(n)), 2 * np.pi * rng.random(n)
    u, v = i * du + rad * np.cos(ang), j * dv + rad * np.sin(ang)
    h = np.zeros(n)
    for cu, cv in 2 * np.pi * rng.random((8, 2)):
        d2 = ((u - cu + np.pi) % (2 * np.pi) - np.pi) ** 2 + ((v - cv + np.pi) % (2 * np.pi) - np.pi) ** 2
        h += 0.009 * np.exp(-d2 / 0.045)
    r = 0.3 + h
    V = np.stack([(1 + r * np.cos(v)) * np.cos(u), (1 + r * np.cos(v)) * np.sin(u), r * np.sin(v)], 1)
    a, b = j * nu + i, j * nu + (i + 1) % nu
    c, d = ((j + 1) % nv) * nu + (i + 1) % nu, ((j + 1) % nv) * nu + i
    F = np.concatenate([np.stack([a, b, c], 1), np.stack([a, c, d], 1)]).astype(np.int32)
    return V, F


def _gen(seed):
    return torch.Generator(device=DEV).manual_seed(seed)


def _randn(g, *shape):
    return torch.randn(*shape, generator=g, device=DEV, dtype=torch.float64)


def _torus_csr(nu, nv, seed):
    """Cotan-like CSR matrix on the torus grid: 7 entries per row, zero row sums."""
    n = nu * nv
    v = torch.arange(n, device=DEV)
    i, j = v % nu, v // nu
    # the six neighbours of the triangulation above, and the vertex itself
    nb = [(di, dj) for di, dj in ((1, 0), (-1, 0), (0, 1), (0, -1), (1, 1), (-1, -1))]
    col = torch.stack([((j + dj) % nv) * nu + (i + di) % nu for di, dj in nb] + [v], 1)
    w = -(0.5 + 0.2 * torch.rand(n, 6, generator=_gen(seed), device=DEV, dtype=torch.float64))
    val = torch.cat([w, -w.sum(1, keepdim=True)], 1)
    col, order = col.sort(1)
    ptr = torch.arange(0, 7 * n + 1, 7, device=DEV, dtype=torch.int32)
    return ptr, col.reshape(-1).to(torch.int32), val.gather(1, order).reshape(-1).contiguous()


def _basis(n, k, seed):
    """Psi (n x k) like an M-orthonormal block and S Psi of the same rows: the
    reduced matrix is near diag(lambda), lambda_j growing linearly (Weyl)."""
    g = _gen(seed)
    Psi = _randn(g, n, k)
    m = 0.8 + 0.4 * torch.rand(n, 1, generator=g, device=DEV, dtype=torch.float64)
    lam = 2.0 * torch.arange(k, device=DEV, dtype=torch.float64) + 0.5
    SP = Psi * m
    SP *= lam / n
    return Psi, SP


def _reduced(k, seed):
    """Reduced matrices after a subspace iteration: unit-diagonal M_bar near I
    and S_bar near diag(lambda), lambda_0 = 0, growing by Weyl's law.  The gaps
    stay open, so that single eigenvectors are well determined."""
    g = _gen(seed)
    gap = 0.5 + torch.rand(k, generator=g, device=DEV, dtype=torch.float64)
    gap[0] = 0.0
    lam = gap.cumsum(0)
    A = torch.eye(k, device=DEV, dtype=torch.float64) + _randn(g, k, k) * (0.1 / k)
    Mb, Sb = A.T @ A, A.T @ (lam[:, None] * A)
    s = Mb.diagonal().rsqrt()
    Mb, Sb = s[:, None] * Mb * s, s[:, None] * Sb * s
    return (0.5 * (Sb + Sb.T)).contiguous(), (0.5 * (Mb + Mb.T)).contiguous()


def _hierarchy(ctx, V, F, p, levels, seed, mixed):
    o = hs.default_options()
    o.levels, o.start_vertex = levels, seed % V.shape[0]
    o.precision = hs.HSIM_MIXED if mixed else hs.HSIM_FP64
    hier = hs.Hierarchy(ctx, F, V=V, p=p, options=o)
    S, M = hs.assemble(ctx, hier, V=torch.as_tensor(V, device=DEV))
    return hier, S, M


def _batch_meshes(case, seed):
    # the sizes belong to the case, the positions to the seed
    rng = np.random.default_rng(1000 * case["count"] + case["p"])
    sizes = np.exp(rng.uniform(np.log(case["lo"]), np.log(case["hi"]), case["count"]))
    # near-square cells: nu : nv as R : r
    grids = [(int(round(math.sqrt(n / 0.3))), int(round(math.sqrt(n * 0.3)))) for n in sizes]
    return [_torus(nu, nv, seed + 1 + i) for i, (nu, nv) in enumerate(grids)]


def _shift(k):
    """A shift inside the lowest part of the spectrum (Weyl on the torus of area
    4 pi^2 R r), as Lambda_floor(alpha p), away from eigenvalues only by chance."""
    return 0.1 * k / 1.5 * 4 * math.pi / (4 * math.pi ** 2 * 0.3) + 0.123


def prepare(case, seed):
    op = case["op"]
    st = {"op": op, "case": case, "ctx": hs.Context(0)}
    if op == "spmm":
        st["ptr"], st["col"], st["val"] = _torus_csr(case["nu"], case["nv"], seed)
        st["X"] = _randn(_gen(seed + 1), case["nu"] * case["nv"], case["k"])[:, case["locked"]:]
    elif op == "gram":
        st["A"], st["B"] = _basis(case["n"], case["k"], seed)
    elif op == "update":
        k = case["k"]
        st["A"] = _randn(_gen(seed), case["n"], k)
        # Ritz vectors: near the identity, columns of unit scale
        st["B"] = torch.eye(k, device=DEV, dtype=torch.float64) + _randn(_gen(seed + 1), k, k) * (0.3 / math.sqrt(k))
    elif op == "ritz":
        st["S"], st["M"] = _reduced(case["k"], seed)
    elif op == "shifted_solve":
        V, F = _torus(case["nu"], case["nv"], seed)
        # a level-0 factorisation: the hierarchy of p eigenpairs, q = k columns
        st["hier"], st["S"], st["M"] = _hierarchy(st["ctx"], V, F, max(1, case["k"] * 2 // 3), 2, seed, case["f32"])
        # the mixed path shifts below the spectrum, the FP64 path into it
        st["mu"] = -_shift(case["k"]) if case["f32"] else _shift(case["k"])
        st["B"] = _randn(_gen(seed), V.shape[0], case["k"]) * st["M"][:, None]
    elif op == "eig_grad":
        V, F = _torus(case["nu"], case["nv"], seed)
        st["V"], st["F"] = torch.as_tensor(V, device=DEV), torch.as_tensor(F, device=DEV)
        st["lam"], st["E"], st["w"] = _modes(case, seed)
    elif op == "solve":
        V, F = _torus(case["nu"], case["nv"], seed)
        st["hier"], st["S"], st["M"] = _hierarchy(st["ctx"], V, F, case["p"], case["levels"], seed, case["mixed"])
    else:
        made = [_hierarchy(st["ctx"], V, F, case["p"], 2, seed + i, True)
                for i, (V, F) in enumerate(_batch_meshes(case, seed))]
        st["hiers"], st["S"], st["M"] = (list(x) for x in zip(*made))
    return st


def _modes(case, seed):
    """p smooth modes cos(a u + b v + c) on the torus grid (column-major, as the
    solve returns them), their Rayleigh quotients by scale, and loss weights."""
    g, p = _gen(seed), case["p"]
    n = case["nu"] * case["nv"]
    i = torch.arange(n, device=DEV, dtype=torch.float64)
    u, v = (i % case["nu"]) * (2 * math.pi / case["nu"]), (i // case["nu"]) * (2 * math.pi / case["nv"])
    a = torch.randint(0, 9, (p, 1), generator=g, device=DEV).double()
    b = torch.randint(0, 4, (p, 1), generator=g, device=DEV).double()
    c = 6.28 * torch.rand(p, 1, generator=g, device=DEV, dtype=torch.float64)
    E = 0.4 * torch.cos(a * u + b * v + c)
    lam = (a * a + b * b / 0.09).reshape(-1) + 0.1
    w = _randn(g, p)
    return lam, E.t(), w


# ---- one pass -------------------------------------------------------------------

def run(st):
    op, c, ctx = st["op"], st["case"], st["ctx"]
    if op == "spmm":
        return hs.spmm(ctx, st["ptr"], st["col"], st["val"], st["X"])
    if op == "gram":
        return hs.gram_tc(ctx, st["A"], st["B"], digits=c["digits"]) if c["tc"] else hs.gram(ctx, st["A"], st["B"])
    if op == "update":
        return (hs.gemm_update_tc if c["tc"] else hs.gemm_update)(ctx, st["A"], st["B"])
    if op == "ritz":
        lam, X, _ = hs.ritz(ctx, st["S"], st["M"], tc=c["tc"])
        return {"lam": lam, "X": _fix_sign(X)}
    if op == "shifted_solve":
        X, neg = hs.shifted_solve(ctx, st["hier"], 0, st["S"], st["M"], st["mu"], st["B"], f32=c["f32"])
        return {"X": X, "negative_pivots": neg}
    if op == "eig_grad":
        return hs.eig_grad(ctx, st["V"], st["F"], st["lam"], st["E"], st["w"])
    if op == "solve":
        lam, Phi, _ = hs.solve(ctx, st["hier"], st["S"], st["M"], c["p"], c["tol"])
        return {"lam": lam, "Phi": Phi}
    out = hs.solve_batched(ctx, st["hiers"], st["S"], st["M"], c["p"], c["tol"])
    return [{"lam": lam, "Phi": Phi} for lam, Phi, _ in out]


def _fix_sign(X):
    """Eigenvectors have no sign of their own: the entry of largest magnitude positive."""
    return X * torch.sign(X.gather(0, X.abs().argmax(0, keepdim=True)))


# ---- what a pass needs, and what it should give ----------------------------------

def _nnz_factor(n):
    # nested dissection of a triangulated surface: about 4.2 n log2 n entries of L
    return 4.2 * n * math.log2(n)


def _solve_work(n, q, p, mixed):
    # two subspace iterations on the finest level at the least: per iteration two
    # solves, one product with S, two Grams (half of each) and the update
    el = 4 if mixed else 8
    flops = 2 * (2 * 4 * _nnz_factor(n) * q + 14.0 * n * q + 4.0 * n * q * q) + 64.0 * n ** 1.5
    byts = 2 * (2 * 2 * el * _nnz_factor(n) + 8 * 8.0 * n * q) + 8.0 * n * (p + 8)
    return byts, flops


def work(case):
    op = case["op"]
    if op == "spmm":
        n, k = case["nu"] * case["nv"], case["k"] - case["locked"]
        return {"bytes": 12.0 * 7 * n + 4 * (n + 1) + 16.0 * n * k, "flops": 14.0 * n * k}
    if op == "gram":
        n, k = case["n"], case["k"]
        return {"bytes": 16.0 * n * k + 8.0 * k * k, "flops": 2.0 * n * k * k}
    if op == "update":
        n, k = case["n"], case["k"]
        return {"bytes": 16.0 * n * k + 8.0 * k * k, "flops": 2.0 * n * k * k}
    if op == "ritz":
        k = case["k"]
        # factor M_bar, reduce, tridiagonalise, transform back twice
        return {"bytes": 24.0 * k * k + 8 * k, "flops": (1 / 3 + 2 + 4 / 3 + 2 + 1) * float(k) ** 3}
    if op == "shifted_solve":
        n, k, el = case["nu"] * case["nv"], case["k"], 4 if case["f32"] else 8
        return {"bytes": 2 * el * _nnz_factor(n) + 16.0 * n * k + 8.0 * 8 * n,
                "flops": 64.0 * n ** 1.5 + 4 * _nnz_factor(n) * k}
    if op == "eig_grad":
        n, p = case["nu"] * case["nv"], case["p"]
        return {"bytes": 8.0 * n * p + 48.0 * n + 24.0 * n, "flops": 2 * n * 12.0 * p}
    if op == "solve":
        b, f = _solve_work(case["nu"] * case["nv"], math.ceil(1.5 * case["p"]), case["p"], case["mixed"])
        return {"bytes": b, "flops": f}
    mean = (case["hi"] - case["lo"]) / math.log(case["hi"] / case["lo"])  # of log-uniform sizes
    b, f = _solve_work(mean, math.ceil(1.5 * case["p"]), case["p"], True)
    return {"bytes": case["count"] * b, "flops": case["count"] * f}


def exact(case, seed):
    op = case["op"]
    if op == "spmm":
        n = case["nu"] * case["nv"]
        _, col, val = _torus_csr(case["nu"], case["nv"], seed)
        X = _randn(_gen(seed + 1), n, case["k"])[:, case["locked"]:]
        col, val, Y = col.view(n, 7).long(), val.view(n, 7), torch.zeros_like(X)
        for t in range(7):
            Y.addcmul_(val[:, t:t + 1], X[col[:, t]])
        return Y
    if op == "gram":
        A, B = _basis(case["n"], case["k"], seed)
        return A.T @ B
    if op == "update":
        k = case["k"]
        B = torch.eye(k, device=DEV, dtype=torch.float64) + _randn(_gen(seed + 1), k, k) * (0.3 / math.sqrt(k))
        return _randn(_gen(seed), case["n"], k) @ B
    if op == "ritz":
        Sb, Mb = (x.cpu() for x in _reduced(case["k"], seed))
        L = torch.linalg.cholesky(Mb)
        T = torch.linalg.solve_triangular(L, Sb, upper=False)
        T = torch.linalg.solve_triangular(L, T.T.contiguous(), upper=False)
        lam, Y = torch.linalg.eigh(0.5 * (T + T.T))
        return {"lam": lam, "X": _fix_sign(torch.linalg.solve_triangular(L.T, Y, upper=True))}
    if op == "shifted_solve" and case["nu"] * case["nv"] <= 20000:
        V, F = _torus(case["nu"], case["nv"], seed)
        S, m = _cotan(torch.as_tensor(V, device=DEV), torch.as_tensor(F, device=DEV).long())
        mu = -_shift(case["k"]) if case["f32"] else _shift(case["k"])
        B = _randn(_gen(seed), V.shape[0], case["k"]) * m[:, None]
        K = S.to_dense()
        K.diagonal().sub_(mu * m)
        return {"X": torch.linalg.solve(K, B), "negative_pivots": None}
    if op == "eig_grad":
        V, F = _torus(case["nu"], case["nv"], seed)
        lam, E, w = _modes(case, seed)
        V, F = torch.as_tensor(V, device=DEV).requires_grad_(), torch.as_tensor(F, device=DEV).long()
        cot, area = _corners(V, F)
        loss = 0.0
        for k in range(3):
            a, b = F[:, (k + 1) % 3], F[:, (k + 2) % 3]
            # phi^T S phi = sum over corners of cot / 2 (phi_a - phi_b)^2
            loss = loss + (0.5 * cot[:, k] * ((E[a] - E[b]) ** 2 @ w)).sum()
            loss = loss - (area / 3 * (E[F[:, k]] ** 2 @ (w * lam))).sum()
        return torch.autograd.grad(loss, V)[0]
    return None


def _corners(V, F):
    """Cotangents of the three corners and the area of each triangle."""
    cot = []
    for k in range(3):
        x, y = V[F[:, (k + 1) % 3]] - V[F[:, k]], V[F[:, (k + 2) % 3]] - V[F[:, k]]
        cross = torch.linalg.cross(x, y).norm(dim=1)
        cot.append((x * y).sum(1) / cross)
    return torch.stack(cot, 1), 0.5 * cross


def _cotan(V, F):
    """Cotan stiffness matrix (sparse) and lumped mass of a mesh."""
    cot, area = _corners(V, F)
    n = V.shape[0]
    m = torch.zeros(n, device=DEV, dtype=torch.float64)
    idx, val = [], []
    for k in range(3):
        m.index_add_(0, F[:, k], area / 3)
        a, b, c = F[:, (k + 1) % 3], F[:, (k + 2) % 3], 0.5 * cot[:, k]
        idx += [torch.stack([a, b]), torch.stack([b, a]), torch.stack([a, a]), torch.stack([b, b])]
        val += [-c, -c, c, c]
    return torch.sparse_coo_tensor(torch.cat(idx, 1), torch.cat(val), (n, n)).coalesce(), m
