"""The GDP phase on shared-memory tiles against the streaming kernel (the general
path), at the edges of what a tile holds: one tile and several, whole and
broken slices, rows of more entries than registers take, tiles too large for
one row a thread, for registers at all, or for the tiles' local indices, every
selection method, phases cut inside a round, traces, long edges."""
import numpy as np
import pytest

import instances as I
import paper_2011_08170_gb300 as f2m
from paper_2011_08170_gb300 import build as B

pytestmark = pytest.mark.gpu
STREAMING, ONE = f2m.F2M_FLAG_STREAMING_GDP, f2m.F2M_FLAG_ONE_SWEEP_GDP


@pytest.fixture(scope="module")
def lib():
    B.build()
    return f2m.load()


def _graph(kind, n, k, seed=1):
    xy = I.uniform_points(n, seed) if kind == "uniform" else I.mixture_points(n, seed)
    return (xy,) + f2m.f2m_knn_csr(xy, k)


def _phase(g, lam0, sweeps, flags=0, b=None, trace=0, **kw):
    ctx = f2m.f2m_create(*g, f2m.f2m_default_params(flags=flags, **kw))
    if b is not None:
        f2m.f2m_set_degrees(ctx, b)
    out = []
    f2m.f2m_set_lambda(ctx, lam0, kw.get("frac_bits", 8))
    for s in sweeps:
        st, sw, tb, tc = f2m.f2m_gdp(ctx, s, trace_cap=trace)
        out.append((st, sw, f2m.f2m_get_lambda(ctx)[0].copy(), None if tb is None else (tb.tolist(), tc.tolist())))
    return out


def _same(a, b):
    for x, y in zip(a, b):
        assert x[:2] == y[:2] and np.array_equal(x[2], y[2]) and x[3] == y[3]


@pytest.mark.parametrize("n", [9, 63, 64, 127, 128, 129, 1000, 4001, 20011])
def test_tiles_equal_streaming(lib, n):
    g = _graph("mixture" if n % 2 else "uniform", n, min(8, n - 1))
    rng = np.random.default_rng(n)
    lam0 = rng.integers(-1 << 20, 1 << 22, size=n).astype(np.int32)
    sweeps = (1, 2, 3, 4, 5, 7, 64)
    want = _phase(g, lam0, sweeps, STREAMING)
    _same(_phase(g, lam0, sweeps), want)
    _same(_phase(g, lam0, sweeps, ONE), want)
    _same(_phase(g, lam0, sweeps, 0, gdp_ctas_per_sm=2), want)
    want = _phase(g, lam0, (5, 30), STREAMING, trace=30)
    _same(_phase(g, lam0, (5, 30), 0, trace=30), want)


@pytest.mark.parametrize("n,k", [(60_000, 10), (130_000, 10), (200_000, 12), (320_000, 8), (700_000, 5), (1_300_000, 4)])
def test_large_tiles_equal_streaming(lib, n, k):
    # 1 and 2 rows a thread; shared-memory entries of 8 and 4 bytes; none fits
    g = _graph("uniform", n, k)
    lam0 = np.zeros(n, np.int32)
    _same(_phase(g, lam0, (1, 6, 33)), _phase(g, lam0, (1, 6, 33), STREAMING))


@pytest.mark.parametrize("bmax", [3, 4, 6, 7, 9])
@pytest.mark.parametrize("n", [500, 30_011])
def test_degree_requirements_equal_streaming(lib, n, bmax):
    g = _graph("uniform", n, 12)
    b = np.random.default_rng(n + bmax).integers(1, bmax + 1, size=n).astype(np.int32)
    lam0 = np.zeros(n, np.int32)
    _same(_phase(g, lam0, (1, 6, 40), b=b), _phase(g, lam0, (1, 6, 40), STREAMING, b=b))


@pytest.mark.parametrize("hub", [17, 40, 254, 255, 400])
def test_deep_rows_equal_streaming(lib, hub):
    # a few nodes adjacent to `hub` others: past the registers' 16 entries, and
    # past the 254 that a slice's depth can say (the streaming kernel takes over)
    n = 3000
    xy, rp, col = _graph("uniform", n, 6)
    rng = np.random.default_rng(hub)
    pairs = {(v, int(c)) for v in range(n) for c in col[rp[v]:rp[v + 1]]}
    for v in (0, 1500, 2999):
        for c in rng.choice(n, hub, replace=False):
            if c != v:
                pairs |= {(v, int(c)), (int(c), v)}
    p = np.array(sorted(pairs))
    rp = np.zeros(n + 1, np.int32)
    rp[1:] = np.cumsum(np.bincount(p[:, 0], minlength=n))
    g = (xy, rp, p[:, 1].astype(np.int32))
    lam0 = np.zeros(n, np.int32)
    _same(_phase(g, lam0, (3, 50)), _phase(g, lam0, (3, 50), STREAMING))


def test_long_edges_and_extreme_lambda(lib):
    # costs above the packed forms' limits, lambda near +-2^29
    rng = np.random.default_rng(3)
    m = (1 << 20) - 1
    xy = np.concatenate([rng.choice([0, m], size=(40, 2)), rng.integers(0, m + 1, size=(360, 2))]).astype(np.int32)
    xy = np.unique(xy, axis=0)
    rp, col = f2m.f2m_knn_csr(xy, 9)
    lam0 = rng.choice([-(1 << 29) + 5, (1 << 29) - 5, 0, 1 << 20], size=len(xy)).astype(np.int32)
    for shift in (1, 2, 8):
        a = _phase((xy, rp, col), lam0, (1, 2, 3, 9), damping_shift=shift)
        _same(a, _phase((xy, rp, col), lam0, (1, 2, 3, 9), STREAMING, damping_shift=shift))
