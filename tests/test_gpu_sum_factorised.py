"""Layout, block shape, persistent grids and tuning of the Cartesian patch
kernels that sum-factorise (2D FP32 of degree 2, 3D FP32 of degree >= 6 and
FP64 of degree 8): the options do not change a bit; and on the parts solved by
products they are accepted and have no effect."""
import pytest

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

import paper_2512_02577_gb300 as p
from paper_2512_02577_gb300.inputs import random_vector
from tests.test_gpu_defaults_high_degree import ctx_default
from tests.test_gpu_parity import to_dev

pytestmark = pytest.mark.gpu
PARTS = [(2, 40, 2, p.FP32), (3, 6, 6, p.FP32), (3, 4, 7, p.FP32), (3, 4, 8, p.FP32), (3, 4, 8, p.FP64)]


def sweeps(d, n, k, prec, smoother, **kw):
    dt = torch.float64 if prec == p.FP64 else torch.float32
    ctx = ctx_default(d, n, k, L=1, prec=prec, smoother=smoother, **kw)
    u = torch.zeros((k * n + 1) ** d, dtype=dt, device="cuda:0")
    ctx.smooth(to_dev(random_vector(d, n, k, seed=901), dt), u, sweeps=2)
    shape = ctx.patch_layout(), ctx.patch_persistent()
    ctx.close()
    return u, shape


@pytest.mark.parametrize("d,n,k,prec", PARTS)
@pytest.mark.parametrize("smoother", [p.ADDITIVE, p.MULTIPLICATIVE])
def test_block_shapes_are_bitwise_equal(d, n, k, prec, smoother):
    ref, shape = sweeps(d, n, k, prec, smoother, patches_per_block=1)
    assert shape[0][0] == p.PATCH_MAJOR and shape[0][1] == 1
    ran = 0
    for kw in (dict(patches_per_block=1, patch_persistent=1), dict(patches_per_block=2), dict(patches_per_block=3),
               dict(patches_per_block=2, patch_persistent=1),
               dict(patch_layout=p.PATCH_INTERLEAVED, patch_threads=128),
               dict(patch_layout=p.PATCH_INTERLEAVED, patch_threads=512, patch_persistent=1)):
        try:
            u, _ = sweeps(d, n, k, prec, smoother, **kw)
        except p.PmgError as e:  # the block does not fit, or the part has no interleaved layout
            assert e.code in (p.PMG_ERR_ARG, p.PMG_ERR_UNSUPPORTED)
            continue
        ran += 1
        assert torch.equal(u, ref), kw
    assert ran >= (1 if k == 8 else 3)


def test_tuned_shape_gives_the_same_sweep():
    d, n, k = 3, 18, 6  # 4,913 patches: the tuner times the candidates
    tuned, shape = sweeps(d, n, k, p.FP32, p.ADDITIVE)
    assert shape[0][0] in (p.PATCH_MAJOR, p.PATCH_INTERLEAVED) and shape[0][1] >= 1
    assert torch.equal(tuned, sweeps(d, n, k, p.FP32, p.ADDITIVE, patches_per_block=1)[0])


@pytest.mark.parametrize("d,n,k,prec", [(3, 6, 4, p.FP32), (3, 4, 7, p.FP64), (2, 20, 3, p.FP32)])
def test_product_parts_take_the_options_without_effect(d, n, k, prec):
    ref, _ = sweeps(d, n, k, prec, p.ADDITIVE)
    u, shape = sweeps(d, n, k, prec, p.ADDITIVE, patches_per_block=2, patch_persistent=1)
    assert shape == ((p.PATCH_MAJOR, 2, shape[0][2]), True)
    assert torch.equal(u, ref)
