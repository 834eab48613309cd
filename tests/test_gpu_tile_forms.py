"""Which kernel and form a GDP phase runs on, as f2m_info.gdp_kernel reports it: the
tiles from 9 points up to what shared memory holds, with one and several sweeps an
exchange, entries whole or packed; the streaming kernel past that and for rows no
tile takes.  (The comparisons of the forms' results with the streaming kernel would
hold for streaming against streaming too.)"""
import math

import numpy as np
import pytest

import instances as I
import paper_2011_08170_gb300 as f2m
from paper_2011_08170_gb300 import build as B

pytestmark = pytest.mark.gpu
STREAMING, ONE, MORE, PACKED = (f2m.F2M_GDP_KERNEL_STREAMING, f2m.F2M_GDP_KERNEL_TILED,
                                f2m.F2M_GDP_KERNEL_TWO_SWEEP, f2m.F2M_GDP_KERNEL_TWO_SWEEP_PACKED)


@pytest.fixture(scope="module")
def lib():
    B.build()
    return f2m.load()


def _ctx(n, k, **kw):
    xy = I.uniform_points(n, 1)
    return f2m.f2m_create(xy, *f2m.f2m_knn_csr(xy, k), f2m.f2m_default_params(max_iters=12, pricing=0, finisher=0, **kw))


def _kernel(ctx):
    return f2m.f2m_solve(ctx, raise_on_error=False).gdp_kernel


@pytest.mark.parametrize("n,k,want", [(9, 5, (MORE,)), (1000, 10, (MORE,)), (20_011, 10, (MORE,)),
                                      (200_000, 12, (PACKED,)), (320_000, 8, (MORE, PACKED)), (700_000, 5, (ONE,)),
                                      (1_300_000, 4, (STREAMING,))])
def test_form_by_size(lib, n, k, want):
    ctx = _ctx(n, k)
    assert _kernel(ctx) in want and _kernel(ctx) in want
    if want != (STREAMING,):
        assert _kernel(_ctx(n, k, flags=f2m.F2M_FLAG_ONE_SWEEP_GDP)) == ONE
    if n <= 320_000:
        assert _kernel(_ctx(n, k, gdp_ctas_per_sm=2)) == ONE
    assert _kernel(_ctx(n, k, flags=f2m.F2M_FLAG_STREAMING_GDP)) == STREAMING


@pytest.mark.parametrize("n", [60_000, 100_000])
def test_the_form_reported_is_the_one_that_ran(lib, n):
    # the first phase guesses rows a thread from the size and runs on that guess if it
    # fits; what the tiles would have needed is known only after it
    own = n // min(152, n // 64)
    rings = {True: 4, False: 3 if own <= 400 else 2}[own <= 200]
    slices = own / 32 + (rings - 1) * ((14 * math.sqrt(own) + 30) / 32 + 1)
    assert slices > 30  # the guess: two rows a thread, packed
    assert _kernel(_ctx(n, 10)) == PACKED


def test_a_first_phase_does_not_try_what_cannot_fit(lib):
    ctx = _ctx(900_000, 8)
    used = []
    for _ in range(2):
        before = f2m.f2m_kernel_launches()
        f2m.f2m_gdp(ctx, 5)
        used.append(f2m.f2m_kernel_launches() - before)
    assert used[0] == used[1]
