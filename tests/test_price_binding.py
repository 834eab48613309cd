"""f2m_price of the binding: one scan where the pairs fit the room it offers, the second
scan's array handed out as it is where they do not (it was copied once more, a quarter
of the call at a million pairs)."""
import ctypes as C

import numpy as np
import pytest

import paper_2011_08170_gb300 as f2m


class _Lib:
    def __init__(self, found):
        self.found, self.into = found, []

    def f2m_price(self, h, cnt, ptr, cap):
        C.cast(cnt, C.POINTER(C.c_int64))[0] = self.found
        self.into.append(ptr)
        if ptr and self.found <= cap:
            a = np.ctypeslib.as_array(C.cast(ptr, C.POINTER(C.c_int32)), (max(self.found, 1), 2))[:self.found]
            a[:] = np.arange(2 * self.found, dtype=np.int32).reshape(-1, 2)
        return 0


class _Ctx:
    n, handle = 1000, 1


@pytest.mark.parametrize("found,scans", [(0, 1), (1, 1), (4096, 1), (4097, 2), (300_000, 2)])
def test_scans_and_copies(monkeypatch, found, scans):
    lib = _Lib(found)
    monkeypatch.setattr(f2m, "load", lambda *a: lib)
    monkeypatch.setattr(f2m, "_check", lambda *a: None)
    c, pairs = f2m.f2m_price(_Ctx())
    assert c == found and pairs.shape == (found, 2) and len(lib.into) == scans
    assert np.array_equal(pairs, np.arange(2 * found, dtype=np.int32).reshape(-1, 2))
    if scans == 2:
        assert pairs.ctypes.data == lib.into[-1]  # no copy
    else:
        assert pairs.base is None and (found == 0 or pairs.ctypes.data != lib.into[0])  # not the room itself
    assert f2m.f2m_price(_Ctx(), cap=found)[0] == found
    if found:
        assert f2m.f2m_price(_Ctx(), cap=found - 1) == (found, None)
