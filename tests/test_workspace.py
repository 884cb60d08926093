"""Device bytes of a Cartesian context besides its vectors: the tables, the
staged products' buffers, and no scratch that only the set-up needs.  No GPU."""
import pytest

import paper_2512_02577_gb300 as p


@pytest.mark.parametrize("k,n,prec,mb", [
    (8, 24, p.FP64, 3),   # table of the cells' operator: 302 tiles x 4 KB and 125 columns of 729 nodes
    (8, 24, p.FP32, 3),
    (7, 24, p.FP32, 2),
    (4, 32, p.FP64, 2),
    (7, 24, p.FP64, 62),  # and the patches': 10 MB, columns of 343 x 2197 nodes, buffers of 76 batches
])
def test_tables_without_set_up_scratch(k, n, prec, mb):
    es = 8 if prec == p.FP64 else 4
    N = (k * n + 1) ** 3
    # level b, u, r; scratch of the operator (and its FP32 copy); CG; patch corrections per colour
    vectors = N * (3 * es + 4 * 8 + (4 * 4 if es == 4 else 0) + 6 * 8 + 8 * es)
    extra = p.bytes_required(p.make_config(dim=3, n_cells=n, degree=k, n_levels=1, mg_precision=prec)) - vectors
    coarse = 2 * 8 * N  # unit vector and operator column of the coarse set-up (one level: the finest)
    assert 0 < extra - coarse < mb * 1e6
