"""Performance cases of the library: what a program that solves Poisson problems with it has it do.

The calls are those of the paper's path and of the benchmark: the matrix-free operator apply (FP64, FP32 and float-float
arithmetic), one vertex-patch smoothing sweep with the local p-multigrid solver, one geometric V-cycle, whole solves
(FP64, and mixed precision as served), and a grouped solve of many small systems; on Cartesian and on smoothly deformed
meshes.  Sizes are those of the benchmark (32^3 Q4, the degree sweep at about 8M DoFs, the deformed 96^3 Q3 mesh, the
served stream of requests) and of the tests.

`exact` states the same operations with dense 1D and patch matrices in 64-bit torch, without the library.
"""
import math

import numpy as np
import torch

import paper_2512_02577_gb300 as pmg

DEV = "cuda:0"
DEFORM_AMP = 0.05
PREC = {"fp64": pmg.FP64, "fp32": pmg.FP32}


def listed():
    return [
        # the smallest problem of the tests and of smoke(): launches and latency of a V-cycle
        {"name": "vcycle_fp64_2d_q2_16", "kind": "vcycle", "dim": 2, "n": 16, "k": 2, "prec": "fp64", "coarse": 64},
        # the operator of the benchmark's headline configuration (the outer iteration's A p)
        {"name": "apply_fp64_q4_32", "kind": "apply", "dim": 3, "n": 32, "k": 4, "prec": "fp64"},
        # the FP32 operator of the degree sweep, an odd mesh of 8M DoFs (residuals of every smoothing step)
        {"name": "apply_fp32_q6_33", "kind": "apply", "dim": 3, "n": 33, "k": 6, "prec": "fp32"},
        # one smoothing sweep of the headline configuration, in the default precision ...
        {"name": "sweep_fp64_q4_32", "kind": "sweep", "dim": 3, "n": 32, "k": 4, "prec": "fp64", "mult": False},
        # ... and in the precision of the mixed solve
        {"name": "sweep_fp32_q4_32", "kind": "sweep", "dim": 3, "n": 32, "k": 4, "prec": "fp32", "mult": False},
        # the degree sweep's high end: an odd mesh, large patches
        {"name": "sweep_fp32_q7_29", "kind": "sweep", "dim": 3, "n": 29, "k": 7, "prec": "fp32", "mult": False},
        # a high-degree sweep in the default precision on a small mesh, the paper's multiplicative smoother
        {"name": "sweep_fp64_q7_12_mult", "kind": "sweep", "dim": 3, "n": 12, "k": 7, "prec": "fp64", "mult": True},
        # the deformed benchmark mesh: stored geometry, bound by memory
        {"name": "apply_fp32_deformed_q3_96", "kind": "apply_def", "n": 96, "k": 3, "prec": "fp32"},
        # one sweep of the deformed smoother
        {"name": "sweep_fp32_deformed_q3_48", "kind": "sweep_def", "n": 48, "k": 3},
        # whole call: the headline solve, FP64 throughout
        {"name": "solve_fp64_q4_32", "kind": "solve", "n": 32, "k": 4, "prec": "fp64", "ff": False, "coarse": 4096},
        # whole call: a large served request, FP32 V-cycle under the float-float operator
        {"name": "solve_mixed_q5_48", "kind": "solve", "n": 48, "k": 5, "prec": "fp32", "ff": True, "coarse": 0},
        # whole call: small served requests solved together
        {"name": "group_mixed_q3_16", "kind": "group", "k": 3, "sizes": "8 4 12 16 8 6 8 16 4 8 12 8 6 8 16 8"},
    ]


def _log_int(rng, lo, hi):
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    kind = rng.choice(["apply", "apply", "sweep", "sweep", "sweep", "apply_def", "sweep_def", "vcycle", "solve", "group"])
    if kind == "apply":
        dim, k = rng.choice([2, 3, 3, 3]), rng.randint(1, 8)
        hi = 200 // k if dim == 3 else 2800 // k
        return {"kind": kind, "dim": dim, "n": _log_int(rng, 4, hi), "k": k, "prec": rng.choice(["fp64", "fp32", "ff"])}
    if kind == "sweep":
        dim, k, prec = rng.choice([2, 3, 3, 3]), rng.randint(2, 7), rng.choice(["fp64", "fp32"])
        hi = (200 if prec == "fp32" else 128) // k if dim == 3 else 1400 // k
        return {"kind": kind, "dim": dim, "n": _log_int(rng, 4, hi), "k": k, "prec": prec, "mult": rng.random() < 0.25}
    if kind == "apply_def":
        return {"kind": kind, "n": _log_int(rng, 8, 96), "k": rng.choice([2, 3]), "prec": rng.choice(["fp32", "fp32", "ff"])}
    if kind == "sweep_def":
        return {"kind": kind, "n": _log_int(rng, 6, 48), "k": rng.choice([2, 3])}
    if kind == "vcycle":
        dim = rng.choice([2, 3])
        n = rng.choice([8, 12, 16, 24, 32, 48, 64]) if dim == 2 else rng.choice([4, 6, 8, 12, 16])
        return {"kind": kind, "dim": dim, "n": n, "k": rng.randint(2, 5), "prec": "fp64", "coarse": rng.choice([0, 512])}
    if kind == "solve":
        prec = rng.choice(["fp64", "fp32", "fp32"])
        n, k = rng.choice([8, 12, 16, 24, 32, 48]), rng.randint(2, 5)
        while n * k > (128 if prec == "fp64" else 240):
            n, k = rng.choice([8, 12, 16, 24, 32, 48]), rng.randint(2, 5)
        return {"kind": kind, "n": n, "k": k, "prec": prec, "ff": prec == "fp32" and rng.random() < 0.5, "coarse": rng.choice([0, 4096])}
    sizes = [rng.choice([4, 6, 8, 8, 8, 12, 16]) for _ in range(rng.randint(2, 16))]
    return {"kind": kind, "k": rng.randint(2, 5), "sizes": " ".join(map(str, sizes))}


# ---------------------------------------------------------------- what a program has in hand before the call
def _nodes(case):
    return [case["k"] * case["n"] + 1] * case.get("dim", 3)


def _vector(shape, gen, dtype=torch.float64):
    """N(0,1) on the free nodes, 0 on the boundary."""
    v = torch.zeros(shape, dtype=dtype, device=DEV)
    inner = v[tuple(slice(1, -1) for _ in shape)]
    inner.copy_(torch.randn(inner.shape, dtype=torch.float64, device=DEV, generator=gen))
    return v


def _inputs(case, seed):
    gen = torch.Generator(device=DEV)
    gen.manual_seed(seed)
    kind = case["kind"]
    if kind == "group":
        return [_vector([case["k"] * n + 1] * 3, gen) for n in map(int, case["sizes"].split())]
    dtype = torch.float32 if case.get("prec") == "fp32" and kind in ("apply", "sweep", "apply_def") or kind == "sweep_def" else torch.float64
    x = [_vector(_nodes(case), gen, dtype)]
    if kind in ("sweep", "sweep_def"):  # right-hand side, and the iterate that the sweep improves
        x.append(0.1 * _vector(_nodes(case), gen, dtype))
    return x


def _config(case, n):
    kind, k = case["kind"], case["k"]
    kw = dict(dim=case.get("dim", 3), n_cells=n, degree=k, coarse_dofs=case.get("coarse", 0))
    if kind in ("apply_def", "sweep_def"):
        kw.update(geometry=pmg.DEFORMED, deform_amp=DEFORM_AMP, n_levels=1)
    if kind in ("apply", "sweep"):
        kw.update(n_levels=1)
    mixed = case.get("prec") == "fp32" or kind in ("sweep_def", "group")
    kw.update(mg_precision=pmg.FP32 if mixed else pmg.FP64)
    if case.get("ff") or case.get("prec") == "ff" or kind == "group":
        kw.update(outer_apply=pmg.APPLY_FLOAT_FLOAT)
    if case.get("mult"):
        kw.update(smoother=pmg.MULTIPLICATIVE)
    return pmg.make_config(**kw)


def prepare(case, seed):
    x = _inputs(case, seed)
    sizes = [int(n) for n in case["sizes"].split()] if case["kind"] == "group" else [case["n"]]
    ctxs = [pmg.Context(_config(case, n), device=DEV) for n in sizes]
    return {"case": case, "ctxs": ctxs, "x": x, "out": [torch.empty_like(v) for v in x]}


def run(state):
    case, ctx, x, out = state["case"], state["ctxs"][0], state["x"], state["out"]
    kind = case["kind"]
    if kind in ("apply", "apply_def"):
        ctx.apply(x[0], out[0], prec=PREC.get(case["prec"], pmg.FP64))
        return out[0]
    if kind in ("sweep", "sweep_def"):
        out[0].copy_(x[1])
        ctx.smooth(x[0], out[0])
        return out[0]
    if kind == "vcycle":
        ctx.vcycle(x[0], out[0])
        return out[0]
    if kind == "solve":
        info = ctx.solve(x[0], out[0], rtol=1e-8, maxit=200)
        return [out[0], info.iterations]
    infos = pmg.solve_group(state["ctxs"], x, out, rtol=1e-8, maxit=200)
    return [out, [i.iterations for i in infos]]


# ---------------------------------------------------------------- the work that a pass cannot do without
def _p_levels(k):
    ps, p = [], 1
    while p < k:
        ps.append(p)
        p = 2 * p + 1
    return ps + [k]


def _apply_work(dim, n, k, es, deformed=False):
    """(bytes, flops) of y = A x: x read, y written (and the stored tensors read); sum factorisation: 2 dim + 1 (3D: 7,
    2D: 4) contractions with the 1D matrices per cell, or twice 2 dim of them around the quadrature points."""
    cells, nodes = n ** dim, (k * n + 1) ** dim
    contraction = 2 * (k + 1) ** (dim + 1)
    if deformed:
        return 2 * nodes * es + cells * 24 * (k + 1) ** 3, cells * (18 * contraction + 15 * (k + 1) ** 3)
    return 2 * nodes * es, cells * (7 if dim == 3 else 4) * contraction


def _local_work(dim, k, deformed=False):
    """flops of one local V-cycle: two vmults per p-level above the first, transfers, two Jacobi steps."""
    f, ps = 1, _p_levels(k)
    for q, p in zip(ps, ps[1:]):
        m, c = 2 * p - 1, 2 * q - 1
        if deformed:
            f += 2 * 2 ** dim * (18 * 2 * (p + 1) ** 4 + 15 * (p + 1) ** 3)
        else:
            f += 2 * (7 if dim == 3 else 4) * 2 * m ** (dim - 1) * (2 * p * p - 1)
        f += 2 * sum(2 * m ** (dim - a) * c ** (a + 1) for a in range(dim)) + 4 * m ** dim
    return f


def _sweep_work(case, n, es, deformed=False):
    dim, k = case.get("dim", 3), case["k"]
    nodes = (k * n + 1) ** dim
    b, f = _apply_work(dim, n, k, es, deformed)
    return b + nodes * es, f * (2 ** dim if case.get("mult") else 1) + (n - 1) ** dim * _local_work(dim, k, deformed)


def _coarsest(case, n, dim):
    """The hierarchy halves while n is even, or until the dense coarse solve takes the mesh."""
    return n % 2 == 1 or (case["k"] * n - 1) ** dim <= case.get("coarse", 0)


def _vcycle_work(case, n, es):
    dim, k = case.get("dim", 3), case["k"]
    f = 0
    m = n
    while not _coarsest(case, m, dim):
        f += 2 * (m - 1) ** dim * _local_work(dim, k) + 2 * _apply_work(dim, m, k, es)[1]
        m //= 2
    return 2 * (k * n + 1) ** dim * es, f + 2 * (k * m - 1) ** (2 * dim)


def work(case):
    kind, k = case["kind"], case["k"]
    es = 4 if case.get("prec") == "fp32" or kind in ("sweep_def", "group") else 8
    if kind in ("apply", "apply_def"):
        b, f = _apply_work(case.get("dim", 3), case["n"], k, es, kind == "apply_def")
    elif kind in ("sweep", "sweep_def"):
        b, f = _sweep_work(case, case["n"], es, kind == "sweep_def")
    elif kind == "vcycle":
        b, f = _vcycle_work(case, case["n"], es)
    else:  # a solve to 1e-8: about 17 iterations of V-cycle, operator and FP64 vector updates
        b = f = 0
        for n in map(int, str(case.get("sizes", case.get("n"))).split()):
            vb, vf = _vcycle_work(case, n, es)
            ab, af = _apply_work(3, n, k, 8)
            b += 17 * (vb + ab + 6 * 8 * (k * n + 1) ** 3)
            f += 17 * (vf + af)
    return {"bytes": b, "flops": f}


# ---------------------------------------------------------------- the same in 64 bits, from dense matrices
def _gauss(n):
    x, w = np.polynomial.legendre.leggauss(n)
    return (x + 1) / 2, w / 2


def _gll(p):
    c = np.zeros(p + 1)
    c[p] = 1
    inner = np.sort(np.polynomial.legendre.legroots(np.polynomial.legendre.legder(c)).real) if p > 1 else []
    for _ in range(3):  # Newton on P_p'
        if p > 1:
            d1, d2 = np.polynomial.legendre.legder(c), np.polynomial.legendre.legder(c, 2)
            inner = inner - np.polynomial.legendre.legval(inner, d1) / np.polynomial.legendre.legval(inner, d2)
    return (np.concatenate([[-1.0], inner, [1.0]]) + 1) / 2


def _lagrange(nodes, x):
    """(values, derivatives) [point, basis function] of the Lagrange basis of `nodes` at x."""
    n = len(nodes)
    V, D = np.ones((len(x), n)), np.zeros((len(x), n))
    for a in range(n):
        for b in range(n):
            if b != a:
                V[:, a] *= (x - nodes[b]) / (nodes[a] - nodes[b])
        for m in range(n):
            if m != a:
                t = np.full(len(x), 1 / (nodes[a] - nodes[m]))
                for b in range(n):
                    if b not in (a, m):
                        t *= (x - nodes[b]) / (nodes[a] - nodes[b])
                D[:, a] += t
    return V, D


def _matrices_1d(p, n):
    """Interior mass and stiffness of degree p on n cells of size 1 (the operator scales by h^(dim-2))."""
    x, w = _gauss(p + 1)
    V, D = _lagrange(_gll(p), x)
    me, ke = V.T @ (w[:, None] * V), D.T @ (w[:, None] * D)
    M, K = np.zeros((p * n + 1,) * 2), np.zeros((p * n + 1,) * 2)
    for c in range(n):
        s = slice(p * c, p * c + p + 1)
        M[s, s] += me
        K[s, s] += ke
    t = lambda a: torch.from_numpy(a[1:-1, 1:-1].copy()).to(DEV)  # noqa: E731
    return t(M), t(K)


def _along(A, x, ax):
    return torch.movedim(torch.tensordot(A, x, dims=([1], [ax])), 0, ax)


def _inner(x):
    return x[tuple(slice(1, -1) for _ in x.shape)].double()


def _pad(x):
    y = torch.zeros([s + 2 for s in x.shape], dtype=x.dtype, device=x.device)
    y[tuple(slice(1, -1) for _ in x.shape)] = x
    return y


def _apply_cart(x, n, k):
    M, K = _matrices_1d(k, n)
    y = 0
    for d in range(x.dim()):
        t = x
        for a in range(x.dim()):
            t = _along(K if a == d else M, t, a)
        y = y + t
    return y * (1.0 / n) ** (x.dim() - 2)


def _kron(ms):
    a = ms[0]
    for b in ms[1:]:
        a = torch.kron(a, b)
    return a


def _interp(p, q):
    """Patch-interior nodes of degree p from those of degree q (each cell's polynomial evaluated at the finer nodes)."""
    V, _ = _lagrange(_gll(q), _gll(p))
    T = np.zeros((2 * p + 1, 2 * q + 1))
    for c in range(2):
        T[p * c: p * c + p + 1, q * c: q * c + q + 1] = V
    return torch.from_numpy(T[1:-1, 1:-1].copy()).to(DEV)


def _damping(dim, p):
    M, K = _matrices_1d(p, 2)
    A = sum(_kron([K if a == d else M for a in range(dim)]) for d in range(dim))
    s = A.diagonal().rsqrt()
    return 4.0 / (3.0 * torch.linalg.eigvalsh((s[:, None] * A * s[None, :]).cpu())[-1].item())


def _local_matrix(dim, k):
    """The local V-cycle on a Cartesian patch (unit scale) as one matrix."""
    B, ps = None, _p_levels(k)
    for i, p in enumerate(ps):
        M, K = _matrices_1d(p, 2)
        A = sum(_kron([K if a == d else M for a in range(dim)]) for d in range(dim))
        if i == 0:
            B = 1.0 / A
            continue
        T = _kron([_interp(p, ps[i - 1])] * dim)
        I = torch.eye(len(A), dtype=A.dtype, device=A.device)
        J = torch.diag(_damping(dim, p) / A.diagonal())
        X = J + T @ (B @ (T.T @ (I - A @ J)))
        B = X + J @ (I - A @ X)
    return B


def _windows(r, k, starts):
    """Patch-interior values of the patches whose first interior vertices are `starts` (per direction)."""
    for a in range(r.dim()):
        idx = (k * starts[a][:, None] + torch.arange(2 * k - 1, device=r.device)[None, :]).reshape(-1)
        r = torch.index_select(r, a, idx)
    shape = [s for a in range(r.dim()) for s in (len(starts[a]), 2 * k - 1)]
    d = r.dim()
    return r.reshape(shape).permute(*range(0, 2 * d, 2), *range(1, 2 * d, 2)).reshape(-1, (2 * k - 1) ** d)


def _scatter(u, z, k, starts):
    d, m = u.dim(), 2 * k - 1
    z = z.reshape([len(s) for s in starts] + [m] * d)
    for off in np.ndindex(*[m] * d):
        at = u
        for a in range(d):  # patches start K nodes apart: a strided slice of u per offset
            st = int(starts[a][1] - starts[a][0]) * k if len(starts[a]) > 1 else 1
            f = int(starts[a][0]) * k + off[a]
            at = torch.movedim(torch.movedim(at, a, 0)[f: f + st * (len(starts[a]) - 1) + 1: st], 0, a)
        at += z[(Ellipsis,) + off]


def _sweep_cart(b, u, n, k, mult, B=None, backward=False):
    dim = b.dim()
    scale = (1.0 / n) ** (dim - 2)
    B = _local_matrix(dim, k) if B is None else B
    if not mult:
        starts = [torch.arange(n - 1, device=b.device)] * dim
        z = _windows(b - _apply_cart(u, n, k), k, starts) @ (B.T * (1.5 / 2 ** dim / scale))
        u = u.clone()
        _scatter(u, z, k, starts)
        return u
    u = u.clone()
    for c in range(2 ** dim):  # vertex parity colours, x the lowest bit; vertex v + 1 of start v
        par = [(c >> (dim - 1 - a)) & 1 for a in range(dim)]
        starts = [torch.arange(0 if q else 1, n - 1, 2, device=b.device) for q in par]
        if all(len(s) for s in starts):
            _scatter(u, _windows(b - _apply_cart(u, n, k), k, starts) @ (B.T / scale), k, starts)
    return u


def _prolong(k, nc):
    """1D embedding of nc coarse cells into 2 nc, interior nodes."""
    nodes = _gll(k)
    P = np.zeros((2 * k * nc + 1, k * nc + 1))
    for c in range(2 * nc):
        V, _ = _lagrange(nodes, (c % 2 + nodes) / 2)
        P[k * c: k * c + k + 1, k * (c // 2): k * (c // 2) + k + 1] = V
    return torch.from_numpy(P[1:-1, 1:-1].copy()).to(DEV)


def _solve_cart(b, n, k):
    """A^-1 b by the generalised eigenvectors of the 1D matrices."""
    M, K = (a.cpu() for a in _matrices_1d(k, n))
    C = torch.linalg.inv(torch.linalg.cholesky(M))
    lam, Q = torch.linalg.eigh(C @ K @ C.T)
    S, lam = (C.T @ Q).to(DEV), lam.to(DEV)  # S^T M S = I, S^T K S = diag(lam)
    x, den = b, 0
    for a in range(b.dim()):
        x = _along(S.T, x, a)
        den = den + lam.reshape([-1 if d == a else 1 for d in range(b.dim())])
    x = x / (den * (1.0 / n) ** (b.dim() - 2))
    for a in range(b.dim()):
        x = _along(S, x, a)
    return x


def _vcycle_cart(b, n, k, B, case):
    if _coarsest(case, n, b.dim()):
        return _solve_cart(b, n, k)
    u = _sweep_cart(b, torch.zeros_like(b), n, k, False, B)
    r = b - _apply_cart(u, n, k)
    P = _prolong(k, n // 2)
    for a in range(b.dim()):
        r = _along(P.T, r, a)
    z = _vcycle_cart(r, n // 2, k, B, case)
    for a in range(b.dim()):
        z = _along(P, z, a)
    return _sweep_cart(b, u + z, n, k, False, B)


class _Deformed:
    """Degree-p operator on the deformed mesh: G_q = w det J J^-1 J^-T at the Gauss points, rounded to FP32."""

    def __init__(self, n, p):
        self.n, self.p, q = n, p, p + 1
        x, w = _gauss(q)
        V, D = (torch.from_numpy(a).to(DEV) for a in _lagrange(_gll(p), x))
        X = ((torch.arange(n, dtype=torch.float64, device=DEV)[:, None] + torch.from_numpy(x).to(DEV)[None]) / n)
        s, c = torch.sin(2 * math.pi * X), 2 * math.pi * torch.cos(2 * math.pi * X)
        f = lambda z, y, xx: DEFORM_AMP * torch.einsum("ai,bj,ck->abcijk", z, y, xx)  # noqa: E731
        g = torch.stack([f(s, s, c), f(s, c, s), f(c, s, s)], -1).reshape(n ** 3, q ** 3, 3)  # gradient of the bump
        h = 1.0 / n
        det = 1 + g.sum(-1)
        # J = h (I + 1 g^T), det J = h^3 det, J^-1 = (I - 1 g^T / det) / h
        W = torch.from_numpy(np.multiply.outer(np.multiply.outer(w, w), w).reshape(-1)).to(DEV)
        r = [e - g / det[..., None] for e in torch.eye(3, dtype=g.dtype, device=DEV)]  # h times the rows of J^-1
        pairs = ((0, 0), (0, 1), (0, 2), (1, 1), (1, 2), (2, 2))
        self.G = [(W * det * h * (r[a] * r[b]).sum(-1)).float().double() for a, b in pairs]
        k3 = lambda a, b, c: torch.kron(torch.kron(a, b), c)  # noqa: E731
        self.grad = [k3(V, V, D), k3(V, D, V), k3(D, V, V)]  # [point, node], x fastest

    def cell(self, u, cells=None):
        """Cell contributions for nodal values u [cell, node]."""
        G = self.G if cells is None else [g[cells] for g in self.G]
        d = [u @ g.T for g in self.grad]
        e = [G[0] * d[0] + G[1] * d[1] + G[2] * d[2], G[1] * d[0] + G[3] * d[1] + G[4] * d[2], G[2] * d[0] + G[4] * d[1] + G[5] * d[2]]
        return e[0] @ self.grad[0] + e[1] @ self.grad[1] + e[2] @ self.grad[2]

    def diagonal(self):
        g = self.grad
        c = [g[0] * g[0], 2 * g[0] * g[1], 2 * g[0] * g[2], g[1] * g[1], 2 * g[1] * g[2], g[2] * g[2]]
        return self.sum(sum(a @ b for a, b in zip(self.G, c)))

    def gather(self, x):
        p, m = self.p, self.p + 1
        return x.unfold(0, m, p).unfold(1, m, p).unfold(2, m, p).reshape(self.n ** 3, m ** 3)

    def sum(self, z):
        n, p, m = self.n, self.p, self.p + 1
        y, z = torch.zeros([p * n + 1] * 3, dtype=z.dtype, device=DEV), z.reshape([n] * 3 + [m] * 3)
        for i, j, l in np.ndindex(m, m, m):
            e = p * (n - 1) + 1
            y[i: i + e: p, j: j + e: p, l: l + e: p] += z[..., i, j, l]
        return y

    def apply(self, x):
        y = torch.zeros_like(x)
        y[1:-1, 1:-1, 1:-1] = self.sum(self.cell(self.gather(x)))[1:-1, 1:-1, 1:-1]
        return y


def _patch_apply(op, d, v):
    """A_j d for patches at cells v + {0, 1}^3, d [patch, m, m, m] on the patch interior."""
    p, n, m = op.p, op.n, 2 * op.p + 1
    x = torch.nn.functional.pad(d, (1, 1) * 3)
    y = torch.zeros_like(x)
    for a, b, c in np.ndindex(2, 2, 2):
        at = (slice(None),) + tuple(slice(p * o, p * o + p + 1) for o in (a, b, c))
        cells = ((v[:, 0] + a) * n + v[:, 1] + b) * n + v[:, 2] + c
        y[at] += op.cell(x[at].reshape(len(d), -1), cells).reshape(len(d), p + 1, p + 1, p + 1)
    return y[:, 1:m - 1, 1:m - 1, 1:m - 1]


def _patch_values(x, p, v):
    """x at the patch-interior nodes of degree p of the patches v."""
    o = torch.arange(1, 2 * p, device=DEV)
    i = [p * v[:, a, None] + o for a in range(3)]
    return x[i[0][:, :, None, None], i[1][:, None, :, None], i[2][:, None, None, :]]


def _local_def(ops, diags, r, v, l):
    p = ops[l].p
    D = _patch_values(diags[l], p, v)
    if l == 0:
        return r / D
    w = _damping(3, p)
    d = w * r / D
    t = r - _patch_apply(ops[l], d, v)
    T = _interp(p, ops[l - 1].p)
    for a in (1, 2, 3):
        t = _along(T.T, t, a)
    z = _local_def(ops, diags, t, v, l - 1)
    for a in (1, 2, 3):
        z = _along(T, z, a)
    d = d + z
    return d + w * (r - _patch_apply(ops[l], d, v)) / D


def _sweep_def(b, u, n, k):
    ops = [_Deformed(n, p) for p in _p_levels(k)]
    diags = [op.diagonal() for op in ops]
    r = b - ops[-1].apply(u)
    z = torch.empty([(n - 1) ** 3] + [2 * k - 1] * 3, dtype=torch.float64, device=DEV)
    g = torch.arange(n - 1, device=DEV)
    v = torch.stack(torch.meshgrid(g, g, g, indexing="ij"), -1).reshape(-1, 3)
    for s in range(0, len(v), 8192):
        w = v[s: s + 8192]
        z[s: s + 8192] = _local_def(ops, diags, _patch_values(r, k, w), w, len(ops) - 1)
    u = u.clone()
    inner = u[1:-1, 1:-1, 1:-1]
    _scatter(inner, z.reshape(len(v), -1) * (1.5 / 8), k, [g] * 3)
    return u


def exact(case, seed):
    x, kind, k = _inputs(case, seed), case["kind"], case["k"]
    if kind == "group":
        return [[_pad(_solve_cart(_inner(b), n, k)) for b, n in zip(x, map(int, case["sizes"].split()))], [None] * len(x)]
    n = case["n"]
    if kind == "apply":
        return _pad(_apply_cart(_inner(x[0]), n, k))
    if kind == "sweep":
        return _pad(_sweep_cart(_inner(x[0]), _inner(x[1]), n, k, case["mult"]))
    if kind == "apply_def":
        return _Deformed(n, k).apply(x[0].double())
    if kind == "sweep_def":
        return _sweep_def(x[0].double(), x[1].double(), n, k)
    if kind == "vcycle":
        return _pad(_vcycle_cart(_inner(x[0]), n, k, _local_matrix(case["dim"], k), case))
    return [_pad(_solve_cart(_inner(x[0]), n, k)), None]
