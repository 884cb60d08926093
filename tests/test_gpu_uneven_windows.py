"""Node by node accuracy of the Cartesian operator and of the local solves when
the values of a cell or patch differ by many orders of magnitude.

Reference: the same operators in extended precision (np.longdouble), from the
oracle's nodes improved by Newton steps.  Bounds, u the unit roundoff:
- operator, FP64: in sum factorisation a result takes three contractions of
  k + 1 products, 3 (k + 2) roundings, of 1D entries that a quadrature of k + 1
  points gives to about 8 (k + 1) roundings each: 27 (k + 2) u of
  (|K| x |M| x |M| + ...) |x|;
- local solve: 1e-12 of |B| |r| in FP64, 2^29 times that in FP32.  The local
  V-cycle in plain FP64 is itself that far off where an entry of B is smallest
  (2.6e3 u at the corners of a patch of k = 8 in 2D)."""
import functools

import numpy as np
import pytest

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

import paper_2512_02577_gb300 as p
from oracle.patch import p_hierarchy
from oracle.quadrature import gauss_legendre, gauss_lobatto_nodes
from tests.test_gpu_defaults_high_degree import ctx_default
from tests.test_gpu_parity import to_dev

pytestmark = pytest.mark.gpu
LD = np.longdouble


def along(A, x, axis):
    return np.moveaxis(np.tensordot(A, x, axes=([1], [axis])), 0, axis)


def legendre(n, x):
    """P_n and its derivative at x."""
    p0, p1, d0, d1 = np.ones_like(x), x.copy(), np.zeros_like(x), np.ones_like(x)
    for i in range(1, n):
        p0, p1, d0, d1 = p1, ((2 * i + 1) * x * p1 - i * p0) / LD(i + 1), d1, d0 + (2 * i + 1) * p1
    return p1, d1


@functools.lru_cache(maxsize=None)
def nodes(k):
    x = 2 * np.asarray(gauss_lobatto_nodes(k), LD) - 1
    for _ in range(3):
        z = x[1:-1]
        P, dP = legendre(k, z)
        x[1:-1] = z - dP * (1 - z * z) / (2 * z * dP - k * (k + 1) * P)
    return (x + 1) / 2


def lagrange(x, at):
    """Values and derivatives [point, basis function] of the Lagrange basis of the nodes x."""
    V, D = np.ones((len(at), len(x)), LD), np.zeros((len(at), len(x)), LD)
    for a in range(len(x)):
        others = [b for b in range(len(x)) if b != a]
        for b in others:
            V[:, a] *= (at - x[b]) / (x[a] - x[b])
        for m in others:
            D[:, a] += np.prod([(at - x[b]) / (x[a] - x[b]) for b in others if b != m] + [np.ones(len(at), LD)],
                               axis=0) / (x[a] - x[m])
    return V, D


@functools.lru_cache(maxsize=None)
def element_1d(k):
    """1D element mass and stiffness on [0, 1]."""
    x = 2 * np.asarray(gauss_legendre(k + 1)[0], LD) - 1
    for _ in range(3):
        P, dP = legendre(k + 1, x)
        x = x - P / dP
    w = 1 / ((1 - x * x) * legendre(k + 1, x)[1] ** 2)
    V, D = lagrange(nodes(k), (x + 1) / 2)
    return V.T @ (w[:, None] * V), D.T @ (w[:, None] * D)


def transfer_1d(q, k):
    """Patch-interior nodes of degree k from those of degree q."""
    T = np.zeros((2 * k + 1, 2 * q + 1), LD)
    for c in range(2):
        T[k * c:k * c + k + 1, q * c:q * c + q + 1] = lagrange(nodes(q), nodes(k))[0]
    return T[1:-1, 1:-1]


def matrices_1d(k, n):
    """Interior 1D mass and stiffness of degree k on n unit cells."""
    me, ke = element_1d(k)
    M, S = np.zeros((k * n + 1,) * 2, LD), np.zeros((k * n + 1,) * 2, LD)
    for c in range(n):
        s = slice(k * c, k * c + k + 1)
        M[s, s] += me
        S[s, s] += ke
    return M[1:-1, 1:-1], S[1:-1, 1:-1]


def tensor_apply(M, S, x):
    y = 0
    for d in range(x.ndim):
        t = x
        for a in range(x.ndim):
            t = along(S if a == d else M, t, a)
        y = y + t
    return y


def uneven(shape, k, seed):
    """Interior vectors (name, values): unit vectors, one large value among N(0,1) ones, a wide range."""
    rng = np.random.default_rng(seed)
    out = []
    for name, at in (("corner", 0), ("mid", k // 2), ("centre", k - 1)):
        at = (at,) * len(shape)
        unit = np.zeros(shape)
        unit[at] = 1.0
        out.append(("unit " + name, unit))
        for big in (30.0, 1e6):
            v = rng.standard_normal(shape)
            v[at] = big
            out.append(("%g %s" % (big, name), v))
    out.append(("wide", rng.standard_normal(shape) * 10.0 ** rng.uniform(-12, 0, shape)))
    out.append(("even", rng.standard_normal(shape)))
    return out


def embed(v, dtype=torch.float64):
    return to_dev(np.pad(v, 1).reshape(-1), dtype)


def interior(t, shape):
    return t.cpu().numpy().astype(LD).reshape([s + 2 for s in shape])[(slice(1, -1),) * len(shape)]


@pytest.mark.parametrize("d,k", [(2, 3), (2, 5), (2, 8), (3, 2), (3, 3), (3, 4), (3, 5), (3, 8)])
def test_operator_is_accurate_node_by_node(d, k):
    n = 2
    ctx = ctx_default(d, n, k, L=1)
    M, S = matrices_1d(k, n)
    shape = (k * n - 1,) * d
    h = LD(1.0 / n) ** (d - 2)
    for name, x in uneven(shape, k, 601 + k):
        y = embed(np.zeros(shape))
        ctx.apply(embed(x), y)
        ref = h * tensor_apply(M, S, x.astype(LD))
        bound = h * tensor_apply(np.abs(M), np.abs(S), np.abs(x).astype(LD))
        err = np.abs(interior(y, shape) - ref)
        assert (err <= 27 * (k + 2) * LD(2.0) ** -53 * bound).all(), (name, float((err / bound).max()))


@functools.lru_cache(maxsize=None)
def local_matrix(d, k, omega, half):
    """Algorithm 3 on one patch (unit scale) as a matrix."""
    def kron(a):
        return functools.reduce(np.kron, a)

    ps = p_hierarchy(k)
    B = None
    for l, q in enumerate(ps):
        M, S = matrices_1d(q, 2)
        A = sum(kron([S if a == e else M for a in range(d)]) for e in range(d))
        if l == 0:
            B = 1 / A
            continue
        T = kron([transfer_1d(ps[l - 1], q)] * d)
        D = LD(omega[l]) / np.diag(A)
        X = np.diag(D) + T @ (B @ (T.T - (T.T @ A) * D[None, :]))
        B = X if half else X + D[:, None] * (np.eye(len(A), dtype=LD) - A @ X)
    return B


@pytest.mark.parametrize("d,k", [(2, 2), (2, 4), (2, 5), (2, 8), (3, 2), (3, 3), (3, 4), (3, 5)])
@pytest.mark.parametrize("prec", [p.FP64, p.FP32])
@pytest.mark.parametrize("smoother,half", [(p.ADDITIVE, 0), (p.ADDITIVE, 1), (p.MULTIPLICATIVE, 0)])
def test_local_solve_is_accurate_node_by_node(d, k, prec, smoother, half):
    dt, tol = (torch.float64, 1e-12) if prec == p.FP64 else (torch.float32, 1e-12 * 2.0 ** 29)
    ctx = ctx_default(d, 2, k, L=1, prec=prec, smoother=smoother, local_half=half)  # one patch
    omega_as, omega = ctx.damping()
    B = local_matrix(d, k, tuple(omega), half) * LD(2.0) ** (d - 2)
    if smoother == p.ADDITIVE:
        B = B * LD(omega_as)
    shape = (2 * k - 1,) * d
    for name, r in uneven(shape, k, 611 + k):
        r = r.astype(np.float64 if prec == p.FP64 else np.float32)
        u = embed(np.zeros(shape), dt)
        ctx.smooth(embed(r, dt), u)
        r = r.astype(LD).reshape(-1)
        err = np.abs(interior(u, shape).reshape(-1) - B @ r)
        bound = np.abs(B) @ np.abs(r)
        assert (err <= tol * bound).all(), (name, float((err / bound).max()))


# the staged products: 27 patches, one uneven window among even ones, against
# the same window with its large value removed and added back
@pytest.mark.parametrize("k", [6, 7])
@pytest.mark.parametrize("smoother", [p.ADDITIVE, p.MULTIPLICATIVE])
def test_staged_local_solves_of_uneven_patches(k, smoother):
    d, n = 3, 4
    ctx = ctx_default(d, n, k, L=1, smoother=smoother)
    shape = (k * n - 1,) * d
    rng = np.random.default_rng(621)
    at = (k + 1, 2 * k + 2, 3 * k - 3)
    even = rng.standard_normal(shape)
    spike = np.zeros(shape)
    spike[at] = 2.0 ** 20
    out = []
    for v in (even, spike, even + spike):
        u = embed(np.zeros(shape))
        ctx.smooth(embed(v), u)
        out.append(interior(u, shape))
    # u is linear in the right-hand side; each of the three is within 1e-12 of its largest value
    scale = [np.abs(o).max() for o in out]
    assert np.abs(out[2] - out[0] - out[1]).max() <= 1e-12 * sum(scale)
