"""Batched GDP on tiles against the streaming batch kernels (the general path):
instances of one tile and several, at the tile's 960 rows, batches of less and of
more than one wave, an instance whose rows no tile takes, caps and fixed points."""
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


def _instances(sizes, k):
    out = []
    for i, n in enumerate(sizes):
        xy = I.uniform_points(n, 70 + i) if i % 2 else I.mixture_points(n, 70 + i)
        out.append((xy,) + f2m.f2m_knn_csr(xy, min(k, n - 1)))
    return out


def _solve(insts, **kw):
    b = f2m.f2m_create_batch(insts, f2m.f2m_default_params(**kw))
    infos, tot = f2m.f2m_solve_batch(b, raise_on_error=False)
    res = []
    for i, f in enumerate(infos):
        r = [f.iterations, f.phases, f.pricing_rounds, f.bound2, f.frac_bits, f.certified, f.status]
        if f.certified:
            lam, fb = f2m.f2m_batch_get_lambda(b, i)
            rp, col, x2 = f2m.f2m_batch_get_x(b, i)
            r += [lam.tobytes(), rp.tobytes(), col.tobytes(), x2.tobytes()]
        res.append(r)
    return tot.gdp_kernel, res


TILES, STREAM = f2m.F2M_GDP_KERNEL_BATCH_TILES, f2m.F2M_GDP_KERNEL_BATCH


# nine points in the square have edges above 2^19, which the tiles' packed
# entries do not hold: that batch streams
@pytest.mark.parametrize("sizes,k,kernel", [((9, 40, 100), 5, STREAM), ((100, 250, 131), 8, TILES),
                                            ((959, 960, 961, 331, 1921), 8, TILES), ((20000, 1000, 7777), 10, TILES),
                                            (tuple(range(3000, 9000, 61)) + (20000,) * 3, 10, TILES)])
def test_tiles_equal_streaming(lib, sizes, k, kernel):
    insts = _instances(sizes, k)
    kern, a = _solve(insts)
    assert kern == kernel
    kern, b = _solve(insts, batch_shape=5)
    assert kern == f2m.F2M_GDP_KERNEL_BATCH
    assert a == b


def test_caps_and_fixed_points(lib):
    insts = _instances((700, 300, 1500), 7)
    for it in (1, 7, 20000):
        assert _solve(insts, max_iters=it)[1] == _solve(insts, max_iters=it, batch_shape=5)[1]


def test_a_row_no_tile_takes(lib):
    # a node adjacent to 255 others: one more than a slice's depth can say, so
    # the batch runs on the streaming kernels (the smallest of whose shapes, which
    # the autotuner tries, take rows of up to 256 entries)
    insts = _instances((900, 1200), 6)
    xy, rp, col = insts[0]
    pairs = {(v, int(c)) for v in range(900) for c in col[rp[v]:rp[v + 1]]}
    more = [c for c in range(1, 900) if (0, c) not in pairs][:255 - int(rp[1])]
    pairs |= {(0, c) for c in more} | {(c, 0) for c in more}
    p = np.array(sorted(pairs))
    rp = np.zeros(901, np.int32)
    rp[1:] = np.cumsum(np.bincount(p[:, 0], minlength=900))
    insts[0] = (xy, rp, p[:, 1].astype(np.int32))
    kern, a = _solve(insts)
    assert kern == f2m.F2M_GDP_KERNEL_BATCH
    assert a == _solve(insts, batch_shape=5)[1]
