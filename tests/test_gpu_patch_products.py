"""Cartesian patch smoother and FP64 apply as products with sector matrices:
partial batches of patches and cells, the smallest meshes, the fixed-point
scaling of the FP64 products and values that are not finite.

Tolerances as in test_gpu_parity (FP64 apply 1e-12, sweep 1e-11, FP32 2e-5).  Scaling the
right-hand side by a power of two is exact in every step, so those results
are compared bit for bit."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

import paper_2512_02577_gb300 as p
from paper_2512_02577_gb300.inputs import random_vector
from tests.parity import rel
from tests.test_gpu_defaults_high_degree import _tol, ctx_default
from oracle import fem
from tests.test_gpu_parity import full, oracle_level, to_dev

pytestmark = pytest.mark.gpu


# patches: 1, 8, 27 in 3D; 1, 16, 17^2 = 18 * 16 + 1 in 2D
@pytest.mark.parametrize("d,n,k", [(3, 2, 1), (3, 2, 2), (3, 3, 3), (3, 2, 5), (3, 4, 5), (3, 2, 4), (3, 2, 6),
                                   (3, 3, 7), (3, 4, 6), (2, 2, 8),
                                   (2, 5, 8), (2, 18, 2), (2, 18, 3), (2, 5, 4), (2, 5, 7), (2, 3, 1)])
@pytest.mark.parametrize("prec", [p.FP64, p.FP32])
@pytest.mark.parametrize("smoother", [p.ADDITIVE, p.MULTIPLICATIVE])
def test_sweep_matches_oracle(d, n, k, prec, smoother):
    dt = torch.float64 if prec == p.FP64 else torch.float32
    ctx = ctx_default(d, n, k, L=1, prec=prec, smoother=smoother)
    fine = oracle_level(d, n, k, "cartesian")
    b, u0 = random_vector(d, n, k, seed=501 + k), random_vector(d, n, k, seed=502 + k)
    u = to_dev(u0, dt)
    ctx.smooth(to_dev(b, dt), u)
    sweep = fine.smooth if smoother == p.ADDITIVE else fine.mult_sweep
    assert rel(u, full(fine, sweep(b[fine.I], u0[fine.I]))) < _tol(prec)


@pytest.mark.parametrize("d,n,k,prec,power", [(3, 4, 4, p.FP64, 900), (3, 4, 4, p.FP64, -900), (2, 6, 2, p.FP64, 600),
                                              (3, 3, 4, p.FP32, 60), (3, 3, 3, p.FP32, -60)])
def test_scaling_by_a_power_of_two_is_exact(d, n, k, prec, power):
    dt = torch.float64 if prec == p.FP64 else torch.float32
    ctx = ctx_default(d, n, k, L=1, prec=prec)
    b = to_dev(random_vector(d, n, k, seed=511), dt)
    s = torch.tensor(2.0 ** power, dtype=dt, device=b.device)
    u, us = torch.zeros_like(b), torch.zeros_like(b)
    ctx.smooth(b, u)
    ctx.smooth(b * s, us)
    assert torch.equal(us, u * s) and float(u.abs().max()) > 0


@pytest.mark.parametrize("prec", [p.FP64, p.FP32])
@pytest.mark.parametrize("value", [float("nan"), float("inf"), -float("inf")])
def test_values_that_are_not_finite_stay_in_their_patches(prec, value):
    # one bad entry strictly inside cell (0, 0, 0): only the patch of vertex (1, 1, 1) holds it
    d, n, k = 3, 4, 3
    dt = torch.float64 if prec == p.FP64 else torch.float32
    ctx = ctx_default(d, n, k, L=1, prec=prec)
    N1 = k * n + 1
    b = to_dev(random_vector(d, n, k, seed=521), dt).reshape(N1, N1, N1)
    clean = torch.zeros_like(b)
    ctx.smooth(b.reshape(-1), clean.reshape(-1))
    b[1, 1, 1] = value
    u = torch.zeros_like(b)
    ctx.smooth(b.reshape(-1), u.reshape(-1))
    inside = torch.zeros_like(b, dtype=torch.bool)
    inside[1:2 * k, 1:2 * k, 1:2 * k] = True
    assert not torch.isfinite(u[inside]).any()
    assert torch.equal(u[~inside], clean[~inside])


def test_zero_right_hand_side_and_extreme_range():
    d, n, k = 3, 3, 4
    ctx = ctx_default(d, n, k, L=1)
    b = torch.zeros((k * n + 1) ** d, dtype=torch.float64, device="cuda:0")
    u = torch.zeros_like(b)
    ctx.smooth(b, u)
    assert not u.any()
    # subnormal residuals: results no further off than the subnormal spacing allows
    r = random_vector(d, n, k, seed=531)
    ctx.smooth(to_dev(r * 2.0 ** -1060), u)
    ref = torch.zeros_like(b)
    ctx.smooth(to_dev(r * 2.0 ** -1060 * 2.0 ** 900), ref)
    assert np.abs(u.cpu().numpy() * 2.0 ** 900 - ref.cpu().numpy()).max() <= 8 * 2.0 ** (-1074 + 900)


# cells: 1, 8, 27 (27 = 16 + 11) in 3D; 1, 16, 25 in 2D; even and odd numbers of nodes per cell
@pytest.mark.parametrize("d,n,k", [(3, 1, 2), (3, 2, 3), (3, 3, 4), (3, 3, 5), (3, 2, 7), (3, 2, 8), (2, 1, 3), (2, 4, 4),
                                   (2, 5, 5), (2, 5, 8), (2, 5, 2)])
def test_fp64_apply_and_residual_match_oracle(d, n, k):
    ctx = ctx_default(d, n, k, L=1)
    m = fem.Mesh(d, n, k)
    A = fem.assemble(m)
    x, b = random_vector(d, n, k, seed=541), random_vector(d, n, k, seed=542)
    ref = fem.apply_full(m, A, x)
    dirty = x + (1.0 - (random_vector(d, n, k, seed=1) != 0)) * 7.0  # boundary entries are ignored
    y, r = to_dev(np.full_like(x, np.nan)), to_dev(np.full_like(x, np.nan))
    ctx.apply(to_dev(dirty), y)
    ctx.residual(to_dev(b), to_dev(dirty), r)
    assert rel(y, ref) < 1e-12 and rel(r, b - ref) < 1e-12
    for power in (800, -800):
        ys = torch.empty_like(y)
        ctx.apply(to_dev(x * 2.0 ** power), ys)
        assert torch.equal(ys, y * 2.0 ** power)


@pytest.mark.parametrize("k,prec", [(6, p.FP64), (7, p.FP64), (5, p.FP64), (6, p.FP32)])
def test_corrections_do_not_depend_on_the_batch(k, prec):
    # 11^3 = 1331 patches: more than one chunk of batches of the staged
    # products; the same values 8 cells further along z (the same parity
    # colours, so the same order of the sum per node) give the same correction
    d, n = 3, 12
    dt = torch.float64 if prec == p.FP64 else torch.float32
    ctx = ctx_default(d, n, k, L=1, prec=prec)
    N1 = k * n + 1
    gen = torch.Generator().manual_seed(551)
    patch = torch.randn((2 * k, 3 * k, 4 * k), generator=gen, dtype=torch.float64).to("cuda:0", dt)
    us = []
    for z in (1, 9):
        b = torch.zeros((N1, N1, N1), dtype=dt, device="cuda:0")
        b[k * z:k * (z + 2), 3 * k:6 * k, 4 * k:8 * k] = patch
        u = torch.zeros_like(b)
        ctx.smooth(b.reshape(-1), u.reshape(-1))
        us.append(u[k * (z - 1):k * (z + 3)].clone())
        assert torch.isfinite(u).all()
    assert us[0].any() and torch.equal(us[0], us[1])
