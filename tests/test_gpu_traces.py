"""Traces of GDP phases on tiles: the streaming kernel's, in each of the tiles' forms
(8- and 4-byte entries, one and two CTAs per SM, every selection of degrees, phases
that end inside a round, at their fixed point or past the trace's end), and what a
trace costs.

The cost: a tile adds two words a sweep, from one warp, while its rows are in shared
memory instead of registers.  The phase's own time with rows in shared memory, per
the kernel's figures, is at most 1.6 times that with rows in registers; the sums are
a warp reduction beside it.  4 times the untraced phase is far from both that and the
thirty times that an atomic of every row took."""
import time

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


def _graph(n, k):
    xy = I.mixture_points(n, 4)
    return (xy,) + f2m.f2m_knn_csr(xy, k)


def _traced(g, sweeps, cap, flags=0, b=None, **kw):
    ctx = f2m.f2m_create(*g, f2m.f2m_default_params(flags=flags, **kw))
    if b is not None:
        f2m.f2m_set_degrees(ctx, b)
    out = []
    for s in sweeps:
        st, sw, tb, tc = f2m.f2m_gdp(ctx, s, trace_cap=cap)
        m = min(sw, cap)
        out.append((st, sw, tb[:m].tolist(), tc[:m].tolist(), f2m.f2m_get_lambda(ctx)[0].tobytes()))
        out.append((f2m.f2m_gdp(ctx, 3)[:2], f2m.f2m_get_lambda(ctx)[0].tobytes()))  # and on, untraced
    return out


@pytest.mark.parametrize("n,k,bmax,kw", [(40, 5, 0, {}), (2000, 10, 0, {}), (20_011, 10, 0, {}), (150_000, 12, 0, {}),
                                         (300_000, 10, 0, {}), (20_011, 10, 0, dict(gdp_ctas_per_sm=2)),
                                         (20_011, 12, 4, {}), (20_011, 12, 7, {}), (3000, 12, 9, {})])
def test_traces_equal_streaming(lib, n, k, bmax, kw):
    g = _graph(n, k)
    b = np.random.default_rng(n).integers(1, bmax + 1, n).astype(np.int32) if bmax else None
    for sweeps, cap in (((1, 2, 5, 12), 20), ((30,), 7)):
        assert _traced(g, sweeps, cap, b=b, **kw) == _traced(g, sweeps, cap, f2m.F2M_FLAG_STREAMING_GDP, b=b)


def test_trace_to_the_fixed_point(lib):
    g = _graph(1500, 8)
    a, b = (_traced(g, (20_000,), 20_000, fl) for fl in (0, f2m.F2M_FLAG_STREAMING_GDP))
    assert a == b and a[0][0] == f2m.F2M_OK and a[0][3][-1] == 0


def test_a_trace_costs_little(lib):
    n = 100_000
    xy = I.uniform_points(n, 1)
    ctx = f2m.f2m_create(xy, *f2m.f2m_knn_csr(xy, 10))
    zero = np.zeros(n, np.int32)

    def us(cap):
        best = 1e9
        for _ in range(6):
            f2m.f2m_set_lambda(ctx, zero, 8)
            t0 = time.perf_counter()
            f2m.f2m_gdp(ctx, 128, trace_cap=cap)  # waits
            best = min(best, time.perf_counter() - t0)
        return best

    us(0)
    plain, traced = us(0), us(128)
    assert traced < 4 * plain, (plain, traced)
