"""Long rows on the tiles: the streaming kernel's sweeps where the warp starts to take
a row together (113 entries; whole slices of such rows), past 254 up to the longest
row a tile takes (1,536) and past it, with several such rows in one slice and in the
rings of other tiles, and the kernel that ran (an instance of 1,000 points or more
with a row of 255 to 1,000 entries had been left to the streaming kernel, at a third
of the speed)."""
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


def _graph(n, k, hubs, length, seed=2):
    xy = I.uniform_points(n, seed)
    rp, col = f2m.f2m_knn_csr(xy, k)
    rng = np.random.default_rng(length)
    src = np.repeat(np.arange(n, dtype=np.int64), np.diff(rp))
    key = [src * n + col]
    for h in hubs:
        have = set(col[rp[h]:rp[h + 1]].tolist()) | {h}
        add = [int(c) for c in rng.permutation(n) if int(c) not in have and int(c) not in hubs][:length - len(have) + 1]
        a = np.array(add, np.int64)
        key += [h * n + a, a * n + h]
    key = np.unique(np.concatenate(key))
    rp = np.zeros(n + 1, np.int32)
    rp[1:] = np.cumsum(np.bincount(key // n, minlength=n))
    assert all(rp[h + 1] - rp[h] == length for h in hubs)
    return xy, rp, (key % n).astype(np.int32)


@pytest.mark.parametrize("n,hubs,length,tiles", [
    (3000, (0,), 255, True), (3000, (5, 1500, 2999), 256, True), (40_000, (7,), 300, True), (2000, (3, 900), 112, True), (2000, (3, 900), 113, True), (2000, tuple(range(40)), 130, True),
    (40_000, (7, 20_000), 500, True), (40_000, (7,), 1000, None), (40_000, (7,), 1200, None), (40_000, (7,), 1535, None), (40_000, (7,), 1536, None),
    (40_000, (7,), 1537, False), (40_000, (7,), 9000, False)])
def test_long_rows_equal_streaming(lib, n, hubs, length, tiles):
    g = _graph(n, 6, hubs, length)
    out = []
    for kw in ({}, dict(flags=f2m.F2M_FLAG_STREAMING_GDP), dict(gdp_ctas_per_sm=2), dict(flags=f2m.F2M_FLAG_ONE_SWEEP_GDP)):
        ctx = f2m.f2m_create(*g, f2m.f2m_default_params(**kw))
        r = []
        for s in (1, 2, 40):
            r.append(f2m.f2m_gdp(ctx, s)[:2] + (f2m.f2m_get_lambda(ctx)[0].tobytes(),))
        st, sw, tb, tc = f2m.f2m_gdp(ctx, 9, trace_cap=9)
        out.append(r + [(st, sw, tb[:sw].tolist(), tc[:sw].tolist())])
    assert all(o == out[0] for o in out)
    info = f2m.solve(*g, params=f2m.f2m_default_params(max_iters=20, pricing=0, finisher=0), raise_on_error=False).info
    if tiles is not None:
        assert (info["gdp_kernel"] != f2m.F2M_GDP_KERNEL_STREAMING) == tiles
