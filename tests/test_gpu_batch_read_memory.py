"""f2m_batch_get_x of a batch on a stream of its own, into pinned and managed arrays:
ready on return, and the arrays of a read-out into pageable ones (integers: equality)."""
import ctypes as C

import numpy as np
import pytest
import torch

import instances as I
import paper_2011_08170_gb300 as f2m
from paper_2011_08170_gb300 import build as B

pytestmark = pytest.mark.gpu


def _managed(count, dtype):
    rt = C.CDLL(f"libcudart.so.{torch.version.cuda.split('.')[0]}")  # torch has loaded it
    p = C.c_void_p()
    size = count * np.dtype(dtype).itemsize
    assert rt.cudaMallocManaged(C.byref(p), C.c_size_t(size), C.c_uint(1)) == 0
    return rt, p, np.frombuffer((C.c_char * size).from_address(p.value), dtype=dtype)


@pytest.mark.parametrize("kind", ["pinned", "managed"])
def test_read_out_on_a_stream(kind):
    B.build()
    L = f2m.load()
    st = torch.cuda.Stream()
    inst = [(lambda d: (d["xy"], d["row_ptr"], d["col"]))(I.make_instance("uniform", n, s, min(10, n - 1)))
            for n, s in ((4, 0), (1500, 2), (3001, 3))]
    b = f2m.f2m_create_batch(inst, stream=st)
    f2m.f2m_solve_batch(b)
    for i in range(len(inst)):
        want = f2m.f2m_batch_get_x(b, i)
        if kind == "pinned":
            out = [torch.zeros(len(a), dtype=t).pin_memory() for a, t in zip(want, (torch.int32, torch.int32, torch.uint8))]
            got, at, held = [o.numpy() for o in out], [o.data_ptr() for o in out], []
        else:
            held = [_managed(len(a), a.dtype) for a in want]
            got, at = [m[2] for m in held], [m[1] for m in held]
        cap = C.c_int64(len(want[1]))
        assert L.f2m_batch_get_x(b.handle, i, C.byref(cap), *at) == f2m.F2M_OK
        for x, y in zip(got, want):
            assert np.array_equal(x, y)
        for rt, p, _ in held:
            rt.cudaFree(p)
    f2m.f2m_destroy_batch(b)
