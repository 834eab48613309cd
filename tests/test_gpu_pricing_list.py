"""The culled scan where its list of block pairs outgrows the room it starts with
(64 a block and 4,096): the pairs of the full scan.

Two nodes in a hundred have a lambda that reaches across the square and all others
one far below zero, so nearly every block pair is listed and the pairs found are
those of the few."""
import numpy as np
import pytest

import instances as I
import paper_2011_08170_gb300 as f2m
from paper_2011_08170_gb300 import build as B

pytestmark = pytest.mark.gpu


def test_an_outgrown_list_is_scanned_whole():
    B.build()
    f2m.load()
    n = 30_000
    xy = I.uniform_points(n, 5)
    rp, col = f2m.f2m_knn_csr(xy, 6)
    rng = np.random.default_rng(5)
    lam = np.full(n, -(1 << 28), np.int32)
    lam[rng.choice(n, n // 50, replace=False)] = 750_000 << 8
    found = []
    for pricing in (1, 2):
        ctx = f2m.f2m_create(xy, rp, col, f2m.f2m_default_params(pricing=pricing))
        f2m.f2m_set_lambda(ctx, lam, 8)
        for _ in range(2):  # the second scan starts with the room
            cnt, pairs = f2m.f2m_price(ctx)
            found.append((cnt, np.unique(pairs, axis=0).tolist()))
    assert found[0][0] > 100_000 and all(f == found[0] for f in found)
