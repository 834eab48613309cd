"""Host memory that outlives a call: finisher work arrays handed from context to
context, batches staged from separate arrays.  Results do not depend on what a
block held before (equality), and sizes that do not fit are refused as before."""
import threading

import numpy as np
import pytest

import instances as I
import paper_2011_08170_gb300 as f2m
from paper_2011_08170_gb300 import build as B

pytestmark = pytest.mark.gpu


def _graph(n, k, seed):
    xy = I.uniform_points(n, seed)
    return (xy,) + f2m.f2m_knn_csr(xy, k)


def _solve(g):
    ctx = f2m.f2m_create(*g)
    info = f2m.f2m_solve(ctx)
    out = [a.copy() for a in f2m.f2m_get_x(ctx)[:3]] + [f2m.f2m_get_lambda(ctx)[0].copy(), info.bound2]
    f2m.f2m_destroy(ctx)
    return out


def _same(a, b):
    return all(np.array_equal(x, y) for x, y in zip(a, b))


def test_work_arrays_from_context_to_context():
    B.build()
    f2m.load()
    graphs = [_graph(n, 8, n) for n in (9000, 500, 3000, 20_000)]
    first = [_solve(g) for g in graphs]
    for i in (3, 1, 0, 2, 3, 2, 1):
        assert _same(_solve(graphs[i]), first[i])
    bad = []

    def work(i):
        for _ in range(4):
            if not _same(_solve(graphs[i]), first[i]):
                bad.append(i)
    threads = [threading.Thread(target=work, args=(i,)) for i in (0, 1, 2, 0)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not bad


def test_batch_parts():
    B.build()
    f2m.load()
    g = [_graph(n, 6, n) for n in (40, 3000, 77)]

    def solve(inst):
        b = f2m.f2m_create_batch(inst)
        f2m.f2m_solve_batch(b)
        out = [a.copy() for i in range(len(inst)) for a in f2m.f2m_batch_get_x(b, i)]
        f2m.f2m_destroy_batch(b)
        return out
    want = solve(g)
    wide = [(np.asfortranarray(x.astype(np.int64)), r.astype(np.int64), np.repeat(c, 2)[::2]) for x, r, c in g]
    assert _same(solve(wide), want)
    x, r, c = g[1]
    for broken in ((x, r, np.append(c, 5000).astype(np.int32)), (x, np.append(r[:-1], -1).astype(np.int32), c)):
        with pytest.raises(f2m.F2MError) as e:
            f2m.f2m_create_batch([g[0], broken, g[2]])
        assert e.value.status == f2m.F2M_ERR_INVALID_ARG
