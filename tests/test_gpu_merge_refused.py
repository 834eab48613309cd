"""f2m_add_edges with a pair that it refuses leaves the graph, x and what follows as
they were: the arrays, a GDP phase on the renumbered graph and a whole solve equal
those of a context that never saw the call."""
import numpy as np
import pytest

import instances as I
import paper_2011_08170_gb300 as f2m
from paper_2011_08170_gb300 import build as B

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("bad", [(-1, 2), (3, 3), (0, 2000)])
@pytest.mark.parametrize("good", [0, 5, 6000])
def test_refused_pairs_change_nothing(bad, good):
    B.build()
    f2m.load()
    n = 2000
    xy = I.uniform_points(n, 3)
    rp, col = f2m.f2m_knn_csr(xy, 5)
    a, b = (f2m.f2m_create(xy, rp, col) for _ in range(2))
    for c in (a, b):
        f2m.f2m_gdp(c, 7)
        f2m.f2m_extract(c)
    rng = np.random.default_rng(good)
    u = rng.integers(0, n // 2, good)
    pairs = np.stack([u, u + 1 + rng.integers(0, n // 2, good)], 1).astype(np.int32)
    with pytest.raises(f2m.F2MError):
        f2m.f2m_add_edges(a, np.concatenate([pairs, np.array([bad], np.int32)]))
    for x, y in zip(f2m.f2m_get_x(a), f2m.f2m_get_x(b)):
        assert np.array_equal(x, y)
    for c in (a, b):
        f2m.f2m_gdp(c, 9)
    assert np.array_equal(f2m.f2m_get_lambda(a)[0], f2m.f2m_get_lambda(b)[0])
    ia, ib = f2m.f2m_solve(a), f2m.f2m_solve(b)
    assert (ia.bound2, ia.certified, ia.nnz) == (ib.bound2, ib.certified, ib.nnz) and ia.certified == 2
    for x, y in zip(f2m.f2m_get_x(a), f2m.f2m_get_x(b)):
        assert np.array_equal(x, y)
