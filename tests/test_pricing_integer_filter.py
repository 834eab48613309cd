"""The pricing scan's integer filter never rejects a pair with z < 0 (host check).

csrc/pricing.cu quantises a tile pair's points and radii in a frame fitted to
its bounding box and lets a pair through when |D|^2 < (R_u + R_v)^2.  This file
evaluates the same quantisation on the CPU (its fp32 operations in numpy
float32) on pairs placed at the boundary z = -1 in frames of every shift, and
checks that each passes, and that every operand of the matrix product stays an
integer that fp16 holds exactly and every partial sum below 2^24.
"""
import math

import numpy as np
import pytest

from test_pricing_filter import boundary_pairs, radius

F32 = np.float32


def frame(box, smax):
    """Shift b of the frame of a bounding box (x0, y0, x1, y1) and largest s."""
    need = max(F32(max(box[2] - box[0], box[3] - box[1])) * F32(1.0 / 2048.0), F32(smax) * F32(1.0 / 1021.0))
    return 0 if need < 1 else int(math.floor(math.log2(float(need)))) + 1


def row(p, s, box, b):
    iq = F32(2.0 ** -b)
    X = int(np.floor(F32(p[0] - box[0]) * iq)) - 1024
    Y = int(np.floor(F32(p[1] - box[1]) * iq)) - 1024
    R = int(np.ceil(F32(F32(s * iq) + F32(0.7075))))
    return X, Y, R, X * X + Y * Y - R * R


@pytest.mark.parametrize("fb", [1, 8, 9])
@pytest.mark.parametrize("spread", [3, 3000, 300000, (1 << 20) - 1])
def test_integer_filter_passes_every_negative_pair(fb, spread):
    rng = np.random.default_rng(77 * fb + spread % 991)
    cases = boundary_pairs(rng, 200, fb, spread)
    assert len(cases) > 100
    for k, (pu, pv, lu, lv) in enumerate(cases):
        su, sv = radius(lu, fb), radius(lv, fb)
        # the pair's own box, widened at random up to the whole square (other points of the tiles)
        grow = [0, 17, 5000, 1 << 20][k % 4]
        box = [max(0, min(pu[0], pv[0]) - int(rng.integers(0, grow + 1))),
               max(0, min(pu[1], pv[1]) - int(rng.integers(0, grow + 1))),
               min((1 << 20) - 1, max(pu[0], pv[0]) + grow), min((1 << 20) - 1, max(pu[1], pv[1]) + grow)]
        b = frame(box, max(su, sv))
        Xu, Yu, Ru, Au = row(pu, su, box, b)
        Xv, Yv, Rv, Av = row(pv, sv, box, b)
        for X, Y, R, A in ((Xu, Yu, Ru, Au), (Xv, Yv, Rv, Av)):
            assert -1024 <= X <= 1023 and -1024 <= Y <= 1023 and 1 <= R <= 1023
            assert all(float(np.float16(v)) == v for v in (A >> 11, A & 2047, -2 * X, -2 * Y, -2 * R))
        terms = [Au >> 11 << 11, Au & 2047, Av >> 11 << 11, Av & 2047, -2 * Xu * Xv, -2 * Yu * Yv, -2 * Ru * Rv]
        assert sum(abs(t) for t in terms) < 1 << 24
        assert sum(terms) == (Xu - Xv) ** 2 + (Yu - Yv) ** 2 - (Ru + Rv) ** 2
        assert sum(terms) < 0, (pu, pv, lu, lv, fb, b)
