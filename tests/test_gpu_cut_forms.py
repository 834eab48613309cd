"""The GDP kernel with cuts at the edges of its forms, against the CPU oracle's
sweeps: bit-exact.

Random labels make long lists: a cut of half the nodes has about a quarter of all
entries in its list, so at 500 points one warp takes it (about 1,000 to 1,400
entries: both sides of the line to the whole block), at 6,500 points its block's
tables (some 18,000 entries of 16 bytes) pass the shared memory and that block
reads global memory while the others keep their tables; many small cuts give a
block many lists of a few entries; eight layers use every bit of the masks; one
node alone is the shortest list.  Lambdas near 2^28 leave the 32-bit range of z.
"""
import numpy as np
import pytest

import instances as I
import paper_2011_08170_gb300 as f2m
from paper_2011_08170_gb300 import build as B

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,k,cuts,big", [
    (300, 6, [1], False),
    (500, 10, [1, 2], False),
    (500, 10, [250, 40, 1, 3, 7, 100, 2, 5], False),
    (1000, 10, [300, 8], True),
    (6500, 10, [1, 900], False),
    (6500, 10, [2], True),
])
def test_cut_sweeps_equal_oracle(oracle_lib, n, k, cuts, big):
    O = oracle_lib
    B.build()
    f2m.load()
    rng = np.random.default_rng(n + len(cuts))
    d = I.make_instance("uniform", n, 11, k)
    rp, col = d["row_ptr"], d["col"]
    cost = O.cost_table(d["xy"], rp, col)
    layers = []
    for m in cuts:
        comp = rng.integers(-1, m, n).astype(np.int32)
        comp[rng.permutation(n)[:m]] = np.arange(m)  # every cut has a node
        layers.append((comp, m))
    lam0 = rng.integers(-(1 << 28), 1 << 28, n) if big else rng.integers(0, 200_000, n)
    lam0 = lam0.astype(np.int32)
    st_o, lam_o, mu_o, it_o, tb_o, tc_o = O.cut_gdp(rp, col, cost, O.Cuts(n, layers), lam0, None, 8, 2, 40, trace=True)
    ctx = f2m.f2m_create(d["xy"], rp, col)
    f2m.f2m_set_lambda(ctx, lam0, 8)
    for comp, m in layers:
        f2m.f2m_add_cut_layer(ctx, comp, m)
    st, sweeps, tb, tc = f2m.f2m_gdp(ctx, 40, trace_cap=40)
    assert sweeps == it_o and (st == f2m.F2M_OK) == (st_o == O.OR_OK)
    assert np.array_equal(f2m.f2m_get_lambda(ctx)[0], lam_o) and np.array_equal(f2m.f2m_get_cut_duals(ctx)[0], mu_o)
    assert np.array_equal(tb[:sweeps], tb_o) and np.array_equal(tc[:sweeps], tc_o)
