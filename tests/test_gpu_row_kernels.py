"""The kernels that walk rows eight lanes at a time and the tiled scan, through
whole solves against the CPU oracle (integers: equality): rows shorter than, as
long as and longer than the lanes, row counts on both sides of a scan tile
(4,096) and of a block's rows, instances of a batch that end inside a warp."""
import numpy as np
import pytest

import instances as I
import paper_2011_08170_gb300 as f2m
from paper_2011_08170_gb300 import build as B
from parity_helpers import compare_solves, same_optimum

pytestmark = pytest.mark.gpu


def _graph(n, k, seed):
    xy = I.uniform_points(n, seed)
    return (xy,) + f2m.f2m_knn_csr(xy, k)


@pytest.mark.parametrize("n,k", [(4, 3), (9, 8), (33, 31), (700, 7), (4096, 5), (4097, 8), (8193, 3)])
def test_solve_equals_oracle(oracle_lib, n, k):
    B.build()
    f2m.load()
    xy, rp, col = _graph(n, k, n + k)
    compare_solves(oracle_lib, f2m, {"xy": xy, "row_ptr": rp, "col": col})


def test_batch_of_small_instances_equals_oracle(oracle_lib):
    B.build()
    f2m.load()
    g = [_graph(n, min(k, n - 1), 7 * n) for n, k in
         ((4, 3), (5, 4), (6, 3), (7, 6), (30, 9), (31, 16), (64, 5), (1001, 10), (4, 3))]
    b = f2m.f2m_create_batch(g)
    infos, _ = f2m.f2m_solve_batch(b)
    for i, q in enumerate(g):
        r = oracle_lib.solve(*q)
        rp, col, x2 = f2m.f2m_batch_get_x(b, i)
        lam, fb = f2m.f2m_batch_get_lambda(b, i)
        assert np.array_equal(rp, r.row_ptr) and np.array_equal(col, r.col)
        assert same_optimum(infos[i].bound2, fb, r.bound2, r.frac_bits)
        assert oracle_lib.certify(q[0], rp, col, x2, lam, fb, infos[i].bound2) == 0
    f2m.f2m_destroy_batch(b)
