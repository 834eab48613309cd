"""Batches in which only some instances fit the tiles: the streaming kernels' results,
whatever the reason (edges past the packed entries, a row past a tile's, more tiles
than the GPU holds), in one wave and in several, over several phases; and the others
stay on the tiles.

That shows in the GDP time: 600 instances of 960 points are two waves on tiles and
stream at over twice that; one more instance that streams alone adds the sweeps of a
few tiles' rows.  The line is at three quarters of all streaming."""
import numpy as np
import pytest

import instances as I
import paper_2011_08170_gb300 as f2m
from paper_2011_08170_gb300 import build as B

pytestmark = pytest.mark.gpu
TILES, STREAM = f2m.F2M_GDP_KERNEL_BATCH_TILES, f2m.F2M_GDP_KERNEL_BATCH


@pytest.fixture(scope="module")
def lib():
    B.build()
    return f2m.load()


def _knn(xy, k):
    return (xy,) + f2m.f2m_knn_csr(xy, k)


def _far(n=12):  # edges across the square
    rng = np.random.default_rng(n)
    return _knn(np.unique(rng.choice([0, (1 << 20) - 1, 5, 9], size=(8 * n, 2)), axis=0)[:n].astype(np.int32), 7)


def _star(n=900, length=255):
    xy, rp, col = _knn(I.uniform_points(n, 7), 6)
    keep = [c for c in np.arange(1, n) if c not in set(col[:rp[1]].tolist())][:length - int(rp[1])]
    key = np.unique(np.concatenate([np.repeat(np.arange(n), np.diff(rp)) * n + col, np.array(keep), np.array(keep) * n]))
    rp = np.zeros(n + 1, np.int32)
    rp[1:] = np.cumsum(np.bincount(key // n, minlength=n))
    assert rp[1] == length
    return xy, rp, (key % n).astype(np.int32)


def _solve(insts, **kw):
    b = f2m.f2m_create_batch(insts, f2m.f2m_default_params(**kw))
    res = []
    for _ in range(2):  # the second solve starts from the first's lambda and graph
        infos, tot = f2m.f2m_solve_batch(b, raise_on_error=False)
        for i, f in enumerate(infos):
            r = [f.iterations, f.phases, f.pricing_rounds, f.bound2, f.frac_bits, f.certified, f.status]
            if f.certified:
                r += [f2m.f2m_batch_get_lambda(b, i)[0].tobytes()] + [a.tobytes() for a in f2m.f2m_batch_get_x(b, i)]
            res.append(r)
    return tot, res


def _some(sizes, k=8):
    return [_knn(I.uniform_points(n, 40 + i) if i % 2 else I.mixture_points(n, 40 + i), min(k, n - 1))
            for i, n in enumerate(sizes)]


@pytest.mark.parametrize("make", [
    lambda: _some((40, 300, 1200)) + [_far()],
    lambda: [_far()] + _some((2500, 961, 960, 17)) + [_star()],
    lambda: _some((20_000,) * 15) + [_far(), _star()] + _some((5000, 400)),
    lambda: _some((300_000, 1500, 700), 6)])
def test_mixed_batches_equal_streaming(lib, make):
    insts = make()
    tot, got = _solve(insts)
    assert tot.gdp_kernel == STREAM
    tot, want = _solve(insts, batch_shape=5)
    assert got == want


def test_the_others_stay_on_tiles(lib):
    base = _some((960,) * 12)
    insts = [base[i % 12] for i in range(600)]
    ms = {}
    for name, batch, kw in (("tiles", insts, {}), ("mixed", insts + [_far()], {}), ("stream", insts, dict(batch_shape=5))):
        for _ in range(3):
            b = f2m.f2m_create_batch(batch, f2m.f2m_default_params(pricing=0, finisher=0, **kw))
            _, tot = f2m.f2m_solve_batch(b, raise_on_error=False)
            ms[name] = min(ms.get(name, 1e9), tot.ms_gdp)
            assert tot.gdp_kernel == (TILES if name == "tiles" else STREAM)
    assert ms["mixed"] < 0.75 * ms["stream"], ms


def test_scratch_does_not_grow_with_the_batch(lib):
    # 6,000 tiles of 200 rows, twenty waves of them.  A wave's scratch is at most 304
    # tiles of 430 KB, 0.13 GB; words, result arenas and the finisher's arrays of 1.2 M
    # nodes and 14 M entries take 0.4 GB more.  All tiles' at once took 1.1 GB.
    import torch
    base = _some((200,) * 12)
    insts = [base[i % 12] for i in range(6000)]
    b = f2m.f2m_create_batch(insts, f2m.f2m_default_params(pricing=0, finisher=0, max_iters=8))
    free = torch.cuda.mem_get_info()[0]
    infos, tot = f2m.f2m_solve_batch(b, raise_on_error=False)
    assert tot.gdp_kernel == TILES
    assert free - torch.cuda.mem_get_info()[0] < 600 << 20
    single = f2m.f2m_create(*base[5], f2m.f2m_default_params(pricing=0, finisher=0, max_iters=8))
    assert infos[5999 // 12 * 12 - 7].iterations == f2m.f2m_solve(single, raise_on_error=False).iterations


def _close(n, count, seed=0):  # points near each other: short edges
    rng = np.random.default_rng(seed)
    return [_knn(np.unique(rng.integers(0, 60_000, (2 * n, 2)), axis=0)[:n].astype(np.int32), 6) for _ in range(count)]


@pytest.mark.parametrize("n,count,extra,want", [
    (40, 300, 0, TILES), (127, 1216, 0, TILES), (127, 1217, 0, STREAM), (128, 1300, 0, TILES), (30, 3000, 2, STREAM),
    (20, 5, 1, STREAM)])
def test_small_instances(lib, n, count, extra, want):
    # 1,216 is four waves of 304 tiles; `extra` larger ones keep their tiles
    base = _close(n, min(count, 20))
    insts = [base[i % len(base)] for i in range(count)] + _some((1500, 700)[:extra])
    if extra == 1:
        insts.append(_far())
    tot, got = _solve(insts)
    assert tot.gdp_kernel == want
    assert got == _solve(insts, batch_shape=5)[1]


def test_many_small_instances_cost_what_they_did(lib):
    # 10,000 instances of 64 points, 33 waves of tiles, take half as long again on tiles
    # as streamed; the line is at a fifth
    base = _close(64, 20)
    insts = [base[i % 20] for i in range(10_000)]

    def ms(shape):
        best = 1e9
        for _ in range(3):
            b = f2m.f2m_create_batch(insts, f2m.f2m_default_params(pricing=0, finisher=0, batch_shape=shape))
            best = min(best, f2m.f2m_solve_batch(b, raise_on_error=False)[1].ms_gdp)
        return best

    default, best = ms(-1), min(ms(shape) for shape in range(12))
    assert default < 1.2 * best, (default, best)
