"""Grouped solves whose patch solves run as staged products (FP64, 3D, degree 6
and 7): bitwise the members' own solves, over one chunk of batches, several,
and levels without patches, and launches that cover all members."""
import pytest

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

import paper_2512_02577_gb300 as p
from tests.test_gpu_grouped import _check_group_equals_solo, _ctx, _rhs

pytestmark = pytest.mark.gpu


# 16^3: 3375 patches, 211 batches (a chunk holds 76); 4^3: 2 batches
@pytest.mark.parametrize("k,ns,kw", [
    (7, (4, 8, 4, 2, 4), dict()),
    (6, (4, 16, 2, 8, 16), dict(local_cycles=2)),
    (6, (8, 4, 2, 4), dict(smoother=p.MULTIPLICATIVE)),
    (7, (4, 8), dict(smoother=p.MULTIPLICATIVE)),
])
def test_grouped_staged_solve_is_bitwise_the_solo_solve(k, ns, kw):
    ctxs = [_ctx(3, n, k, **kw) for n in ns]
    bs = [_rhs(3, n, k, 700 + i) for i, n in enumerate(ns)]
    infos, _ = _check_group_equals_solo(ctxs, bs)
    assert all(i.status == 0 and i.rel_residual <= 1e-8 for i in infos)
    for c in ctxs:
        c.close()


@pytest.mark.parametrize("k", [6, 7])
def test_grouped_staged_launches_cover_all_members(k):
    # equal systems (so equal iterations): eight of them launch no more than two,
    # but for the residual copies (one per system, iteration and start)
    n = 4
    launches = []
    for m in (2, 8):
        ctxs = [_ctx(3, n, k) for _ in range(m)]
        bs = [_rhs(3, n, k, 710) for _ in range(m)]
        infos, count = _check_group_equals_solo(ctxs, bs)
        launches.append(count)
        for c in ctxs:
            c.close()
    assert launches[1] <= launches[0] + 6 * (infos[0].iterations + 2)
