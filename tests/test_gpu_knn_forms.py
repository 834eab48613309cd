"""The k-NN kernel and the candidate graph at the edges of their forms, against the
CPU oracle (integers: equality): list lengths on both sides of each kernel's,
squares that start too small or too large (far points, tight clusters, lattices
whose distances tie), hub rows too long to be ordered by counting, keys wider
than 64 bits; the warm-start features against the 64-bit formula, bit for bit."""
import numpy as np
import pytest

import instances as I
import oracle
import paper_2011_08170_gb300 as f2m
from paper_2011_08170_gb300 import build as B

pytestmark = pytest.mark.gpu
TOP = (1 << 20) - 1


def _points(kind):
    rng = np.random.default_rng(5)
    if kind == "uniform":
        return I.uniform_points(2000, 3)
    if kind == "cluster and far points":
        a = rng.integers(500_000, 500_040, size=(900, 2))
        b = np.array([(0, 0), (TOP, TOP), (0, TOP), (TOP, 0), (7, 9), (TOP, 500_000)])
        return np.concatenate([a, b]).astype(np.int32)
    if kind == "lattice":
        g = np.arange(0, 40) * 26_000
        return np.stack(np.meshgrid(g, g), -1).reshape(-1, 2).astype(np.int32)
    if kind == "line":
        x = np.unique(rng.integers(0, TOP, 700))
        return np.stack([x, np.full_like(x, TOP)], 1).astype(np.int32)
    pts = np.full((1500, 2), 77_777, np.int32)  # copies: the first k + 1 list and are listed by all
    pts[1400:] = I.uniform_points(100, 8)
    return pts


@pytest.fixture(scope="module")
def lib():
    B.build()
    return f2m.load()


@pytest.mark.parametrize("kind", ["uniform", "cluster and far points", "lattice", "line", "copies"])
@pytest.mark.parametrize("k", [1, 8, 9, 10, 11, 12, 13, 16, 17, 32])
def test_lists_and_graph_equal_oracle(lib, oracle_lib, kind, k):
    xy = _points(kind)
    nbr, d2 = f2m.f2m_knn(xy, k)
    onbr, od2 = oracle.knn(xy, k)
    assert np.array_equal(d2, od2) and np.array_equal(nbr, onbr)
    rp, col = f2m.f2m_knn_csr(xy, k)
    orp, ocol = oracle.knn_csr(xy, k)
    assert np.array_equal(rp, orp) and np.array_equal(col, ocol)


def test_wide_keys(lib):
    n = (1 << 23) + 11
    xy = np.random.default_rng(1).integers(0, TOP + 1, size=(n, 2)).astype(np.int32)
    xy[-1] = xy[0]  # a copy: the smaller index comes first
    nbr, d2 = f2m.f2m_knn(xy, 3)
    for i in (0, 1, 12_345, 1 << 22, n - 2, n - 1):
        d = ((xy.astype(np.int64) - xy[i]) ** 2).sum(1)
        d[i] = 1 << 62
        near = np.lexsort((np.arange(n), d))[:3] if i < 1 else np.argpartition(d, 64)[:64]
        near = near[np.lexsort((near, d[near]))][:3]
        assert np.array_equal(nbr[i], near) and np.array_equal(d2[i], d[near])


@pytest.mark.parametrize("kind", ["uniform", "cluster and far points", "lattice", "line", "copies"])
def test_features_are_the_64_bit_ones(lib, oracle_lib, kind):
    xy = _points(kind)
    if kind == "uniform":
        xy = I.mixture_points(60_000, 4)
    feat, scale = f2m.f2m_features(xy)
    d = np.sqrt(f2m.f2m_knn(xy, 16)[1].astype(np.float64))
    s = np.zeros(len(xy))
    for j in range(16):  # in this order
        s += d[:, j]
    s = np.maximum(1.0, s / 16)
    assert np.array_equal(scale, s.astype(np.float32))
    assert np.array_equal(feat, (d / s[:, None]).astype(np.float32))


def test_features_into_any_float(lib):
    import torch
    xy = I.uniform_points(500, 6)
    feat, scale = f2m.f2m_features(xy)
    d = torch.from_numpy(xy).cuda()
    f, s = torch.zeros(500 * 16 + 3, device="cuda"), torch.zeros(501, device="cuda")
    for o in (0, 1, 2, 3):
        assert lib.f2m_features(d.data_ptr(), 500, f[o:].data_ptr(), s[1:].data_ptr(), None) == f2m.F2M_OK
        assert np.array_equal(f[o:o + 8000].cpu().numpy().reshape(500, 16), feat)
        assert np.array_equal(s[1:].cpu().numpy(), scale)
