"""The FP64 Cartesian operator on both sides of the line between line passes and
cell products (3D, degree 8: up to 8^3 cells by lines), alone and in a grouped
solve with members on either side, against the line passes of the
allocation-free entry point."""
import pytest

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

import paper_2512_02577_gb300 as p
from paper_2512_02577_gb300.inputs import random_vector
from tests.parity import rel
from tests.test_gpu_defaults_high_degree import ctx_default
from tests.test_gpu_grouped import _check_group_equals_solo, _ctx, _rhs
from tests.test_gpu_parity import to_dev

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [8, 9, 10])
def test_degree_8_apply_matches_line_passes(n):
    d, k = 3, 8
    ctx = ctx_default(d, n, k, L=1, prec=p.FP32)
    x = to_dev(random_vector(d, n, k, seed=801))
    y, ref = torch.empty_like(x), torch.empty_like(x)
    ctx.apply(x, y)
    p.apply_cartesian_noalloc(d, n, k, x, ref)
    torch.cuda.synchronize()
    # 27 (k + 2) roundings of |A||x|, an order above |A x|
    assert rel(y, ref) < 1e-12


def test_degree_8_group_with_members_on_both_sides():
    ns = (16, 4, 8)
    ctxs = [_ctx(3, n, 8, mg_precision=p.FP32) for n in ns]
    bs = [_rhs(3, n, 8, 810 + i) for i, n in enumerate(ns)]
    infos, _ = _check_group_equals_solo(ctxs, bs)
    assert all(i.status == 0 and i.rel_residual <= 1e-8 for i in infos)
    for c in ctxs:
        c.close()
