"""f2m_create_batch_parts where no memory can be pinned (here: no GPU at all): the call
goes on with pageable memory, to where the union is put on the device."""
import numpy as np
import pytest

import paper_2011_08170_gb300 as f2m
from paper_2011_08170_gb300 import build as B


def test_staging_does_not_need_pinned_memory():
    import torch
    if torch.cuda.is_available():
        pytest.skip("memory can be pinned here")
    B.build()
    f2m.load()
    xy = np.array([[0, 0], [3, 0], [0, 4], [5, 5], [9, 1]], np.int32)
    rp = np.arange(0, 21, 4, dtype=np.int32)
    col = np.array([[c for c in range(5) if c != v] for v in range(5)], np.int32).ravel()
    with pytest.raises(f2m.F2MError) as e:
        f2m.f2m_create_batch_parts([[xy, rp, col]] * 2)
    assert "staging" not in str(e.value) and "row_ptr" in str(e.value)


@pytest.mark.parametrize("bad", [
    lambda x, r, c: (x, r, c[:-1]),                      # fewer columns than the offsets say
    lambda x, r, c: (x[:-1], r, c),
    lambda x, r, c: (x, r, c.astype(np.int64)),
    lambda x, r, c: (x, np.repeat(r, 2)[::2], c),        # not contiguous
    lambda x, r, c: (x, r[:1], c),
    lambda x, r, c: (x, r.tolist(), c)])
def test_parts_that_do_not_fit_are_refused(bad):
    B.build()
    xy = np.array([[0, 0], [3, 0], [0, 4], [5, 5], [9, 1]], np.int32)
    rp = np.arange(0, 21, 4, dtype=np.int32)
    col = np.array([[c for c in range(5) if c != v] for v in range(5)], np.int32).ravel()
    with pytest.raises(ValueError):
        f2m.f2m_create_batch_parts([(xy, rp, col), bad(xy, rp, col)])


def test_small_instances_are_joined_here(monkeypatch):
    # per-array calls made a batch of 20,000 small instances five times slower to create
    B.build()
    xy = np.array([[0, 0], [3, 0], [0, 4], [5, 5], [9, 1]], np.int32)
    rp = np.arange(0, 21, 4, dtype=np.int32)
    col = np.array([[c for c in range(5) if c != v] for v in range(5)], np.int32).ravel()
    big_rp = np.arange(0, 8193, 8, dtype=np.int32)
    big = (np.zeros((1024, 2), np.int32), big_rp, np.zeros(8192, np.int32))
    seen = []

    class Lib:
        def f2m_create_batch(self, *a):
            seen.append("joined")
            return 1

        def f2m_create_batch_parts(self, *a):
            seen.append("parts")
            return 1

        def f2m_status_string(self, st):
            return b"x"

        def f2m_last_error(self, c):
            return b"y"

    monkeypatch.setattr(f2m, "load", lambda *a: Lib())
    for insts in ([(xy, rp, col)] * 3, [big] * 2, [big, (xy, rp, col)], [(xy.tolist(), rp.tolist(), col.tolist())],
                  [(big[0], big_rp, big[2][:-1])]):
        with pytest.raises(f2m.F2MError):
            f2m.f2m_create_batch(insts)
    assert seen == ["joined", "parts", "parts", "joined", "joined"]
