"""The forms of the pricing scan find the same pairs: all tile pairs (small and
large tiles), the culled list, and the oracle's double loop, at the edges of the
128-point blocks, with radii from none to the whole square."""
import numpy as np
import pytest

import instances as I
import paper_2011_08170_gb300 as f2m
from paper_2011_08170_gb300 import build as B

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def lib():
    B.build()
    return f2m.load()


def _scan(xy, rp, col, lam, pricing, fb=8):
    ctx = f2m.f2m_create(xy, rp, col, f2m.f2m_default_params(pricing=pricing))
    f2m.f2m_set_lambda(ctx, lam, fb)
    cnt, p = f2m.f2m_price(ctx)
    assert cnt == len(p)
    return p[np.lexsort((p[:, 1], p[:, 0]))]


@pytest.mark.parametrize("n", [9, 127, 128, 129, 257, 1000, 2049])
@pytest.mark.parametrize("kind", ["uniform", "mixture"])
def test_forms_equal_the_oracle(lib, oracle_lib, n, kind):
    d = I.make_instance(kind, n, n, 4)
    xy, rp, col = d["xy"], d["row_ptr"], d["col"]
    rng = np.random.default_rng(n)
    spacing = 1e6 / np.sqrt(n)
    for scale in (0.2, 0.6, 20.0):  # few pairs, some, most
        lam = (rng.uniform(-0.3, 1.0, size=n) * scale * spacing * 256).astype(np.int64)
        lam = np.clip(lam, -(1 << 29) + 1, (1 << 29) - 1).astype(np.int32)
        cnt, want = oracle_lib.pricing(xy, rp, col, lam, 8)
        for pricing in (1, 2):
            assert np.array_equal(_scan(xy, rp, col, lam, pricing), want), (scale, pricing)


@pytest.mark.parametrize("kind", ["uniform", "mixture"])
def test_large_tiles_equal_the_oracle_and_the_other_forms(lib, oracle_lib, kind):
    # 60,013 points: more large tiles than the rule asks for; the outlier's
    # radius is larger than a block
    n = 60013
    xy = I.uniform_points(n, 5) if kind == "uniform" else I.mixture_points(n, 5)
    rp, col = f2m.f2m_knn_csr(xy, 8)
    rng = np.random.default_rng(5)
    lam = rng.integers(-100 << 8, 1900 << 8, size=n).astype(np.int32)
    lam[rng.integers(0, n, size=3)] = 40000 << 8
    cnt, want = oracle_lib.pricing(xy, rp, col, lam, 8)
    assert cnt > 0
    a = _scan(xy, rp, col, lam, 1)
    b = _scan(xy, rp, col, lam, 2)
    ctx = f2m.f2m_create(xy, rp, col, f2m.f2m_default_params(flags=f2m.F2M_FLAG_PRICING_TENSOR))
    f2m.f2m_set_lambda(ctx, lam, 8)
    _, c = f2m.f2m_price(ctx)
    c = c[np.lexsort((c[:, 1], c[:, 0]))]
    assert np.array_equal(a, want) and np.array_equal(b, want) and np.array_equal(c, want)
