"""f2m_batch_get_x into host and device arrays, all and some of them: the same
arrays each way, equal to a single solve's (integers: equality)."""
import ctypes as C

import numpy as np
import pytest
import torch

import instances as I
import paper_2011_08170_gb300 as f2m
from paper_2011_08170_gb300 import build as B

pytestmark = pytest.mark.gpu


def test_batch_read_out_host_and_device():
    B.build()
    L = f2m.load()
    inst = []
    for n, seed in ((4, 0), (40, 1), (1500, 2), (257, 3)):
        d = I.make_instance("uniform", n, seed, min(10, n - 1))
        inst.append((d["xy"], d["row_ptr"], d["col"]))
    b = f2m.f2m_create_batch(inst)
    f2m.f2m_solve_batch(b)
    for i, g in enumerate(inst):
        rp, col, x2 = f2m.f2m_batch_get_x(b, i)  # host arrays
        ctx = f2m.f2m_create(*g)
        f2m.f2m_solve(ctx)
        srp, scol, sx2, _ = f2m.f2m_get_x(ctx)
        assert np.array_equal(rp, srp) and np.array_equal(col, scol) and np.array_equal(x2, sx2)
        m = len(col)
        # an odd byte offset into the x array: bytes have no alignment to keep
        dev = (torch.zeros(len(rp) + 1, dtype=torch.int32, device="cuda")[1:],
               torch.zeros(m + 1, dtype=torch.int32, device="cuda")[1:],
               torch.zeros(m + 1, dtype=torch.uint8, device="cuda")[1:])
        out = f2m.f2m_batch_get_x(b, i, out=dev)
        for a, want in zip(out, (rp, col, x2)):
            assert np.array_equal(a.cpu().numpy(), want)
        # columns to the host, x to the device, no row offsets
        hc, dx = np.zeros(m, np.int32), torch.zeros(m, dtype=torch.uint8, device="cuda")
        cap = C.c_int64(m)
        assert L.f2m_batch_get_x(b.handle, i, C.byref(cap), None, hc.ctypes.data, dx.data_ptr()) == f2m.F2M_OK
        assert np.array_equal(hc, col) and np.array_equal(dx.cpu().numpy(), x2)
    f2m.f2m_destroy_batch(b)
