"""Sweeps with cuts on the longest edges the coordinates allow, against the CPU oracle:
bit-exact.  The kernel keeps z in 32 bits where the duals are small, trusting that
a cost in units 2^-F stays below 2^29; blocks read their tables only when all of
their warps have written them, so several runs agree."""
import numpy as np
import pytest

import paper_2011_08170_gb300 as f2m
from paper_2011_08170_gb300 import build as B

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,cuts", [(40, [3]), (700, [5, 60]), (4000, [2, 300, 1])])
def test_longest_edges_equal_oracle(oracle_lib, n, cuts):
    O = oracle_lib
    B.build()
    f2m.load()
    m = (1 << 20) - 1
    rng = np.random.default_rng(n)
    # points on the border of the square, and candidates between random ones
    t = rng.integers(0, m + 1, n)
    side = np.arange(n) % 4
    xy = np.stack([np.where(side < 2, t, np.where(side == 2, 0, m)), np.where(side < 2, side * m, t)], 1)
    xy[:4] = [[0, 0], [m, m], [0, m], [m, 0]]
    xy = xy.astype(np.int32)
    pairs = {(0, 1), (2, 3)} | {(v, (v + d) % n) for v in range(n) for d in (1, 2, 7)}
    for a, b in rng.integers(0, n, (6 * n, 2)):
        if a != b:
            pairs.add((int(a), int(b)))
    key = np.unique([a * n + b for p in pairs for a, b in (p, p[::-1])])
    rp = np.zeros(n + 1, np.int32)
    rp[1:] = np.cumsum(np.bincount(key // n, minlength=n))
    col = (key % n).astype(np.int32)
    cost = O.cost_table(xy, rp, col)
    assert cost.max() > 1_482_000
    layers = []
    for c in cuts:
        comp = rng.integers(-1, c, n).astype(np.int32)
        comp[rng.permutation(n)[:c]] = np.arange(c)
        layers.append((comp, c))
    lam0 = rng.integers(0, 1 << 22, n).astype(np.int32)
    st_o, lam_o, mu_o, it_o, tb_o, tc_o = O.cut_gdp(rp, col, cost, O.Cuts(n, layers), lam0, None, 8, 2, 30, trace=True)
    for _ in range(5):
        ctx = f2m.f2m_create(xy, rp, col)
        f2m.f2m_set_lambda(ctx, lam0, 8)
        for comp, c in layers:
            f2m.f2m_add_cut_layer(ctx, comp, c)
        st, sweeps, tb, tc = f2m.f2m_gdp(ctx, 30, trace_cap=30)
        assert sweeps == it_o and (st == f2m.F2M_OK) == (st_o == O.OR_OK)
        assert np.array_equal(f2m.f2m_get_lambda(ctx)[0], lam_o)
        assert np.array_equal(f2m.f2m_get_cut_duals(ctx)[0], mu_o)
        assert np.array_equal(tb[:sweeps], tb_o) and np.array_equal(tc[:sweeps], tc_o)
