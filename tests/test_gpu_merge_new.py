"""The merge of a scan's pairs (distinct, outside the graph, nothing read back)
against the general merge of the same pairs: the same rows, columns and costs,
and the same GDP phase on the renumbered graph; row counts on both sides of a
scan tile, rows that gain nothing, one, and dozens of columns."""
import numpy as np
import pytest

import instances as I
import paper_2011_08170_gb300 as f2m
from paper_2011_08170_gb300 import build as B

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,k,raise_,hub", [(9, 3, 400_000, 0), (700, 4, 200_000, 0), (4096, 3, 60_000, 500), (4097, 5, 100_000, 0),
                                            (9000, 6, 60_000, 300)])
def test_solve_merges_equal_added_edges(n, k, raise_, hub):
    B.build()
    f2m.load()
    xy = I.uniform_points(n, n)
    rp, col = f2m.f2m_knn_csr(xy, k)
    rng = np.random.default_rng(n)
    lam = rng.integers(0, raise_ << 8, n).astype(np.int32)
    if hub:  # one node whose lambda reaches far
        lam[hub] = 150_000 << 8
    # no sweeps: the solve prices this lambda, merges, and stops at the pricing limit
    a = f2m.f2m_create(xy, rp, col, f2m.f2m_default_params(max_iters=1, finisher=0, max_pricing_rounds=1))
    f2m.f2m_set_lambda(a, lam, 8)
    i = f2m.f2m_solve(a, raise_on_error=False)
    lam1 = f2m.f2m_get_lambda(a)[0].copy()
    got = [x.copy() for x in f2m.f2m_get_x(a)]
    b = f2m.f2m_create(xy, rp, col, f2m.f2m_default_params(max_iters=1, finisher=0))
    f2m.f2m_set_lambda(b, lam, 8)
    f2m.f2m_gdp(b, 1)
    m, pairs = f2m.f2m_price(b)
    assert m == i.edges_added > 0
    pairs = pairs[rng.permutation(m)]
    f2m.f2m_add_edges(b, np.concatenate([pairs, pairs[:3, ::-1]]))  # the general merge drops copies
    want = f2m.f2m_get_x(b)
    for x, y in ((got[0], want[0]), (got[1], want[1]), (got[3], want[3])):
        assert np.array_equal(x, y)
    f2m.f2m_set_lambda(a, lam1, 8)
    f2m.f2m_set_lambda(b, lam1, 8)
    f2m.f2m_gdp(a, 5)
    f2m.f2m_gdp(b, 5)
    assert np.array_equal(f2m.f2m_get_lambda(a)[0], f2m.f2m_get_lambda(b)[0])
