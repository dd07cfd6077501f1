"""Limits of the traveltime call: what it refuses before anything reaches the
device."""
import ctypes as C

import numpy as np
import pytest

from paper_2001_06444_gb300 import rtm

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def test_more_problems_than_32_bits_count_are_refused():
    # a problem's index is a 32-bit integer in the kernels: 2^31 of them would
    # write iterations, times and fields in front of their arrays
    ns, nsrc = 1 << 16, 1 << 15
    vel = torch.full((ns, 1, 1), 2000.0, device="cuda")
    src, rec = np.zeros(nsrc, np.int32), np.zeros(1, np.int32)
    out = torch.full((16,), -7.0, device="cuda")
    with rtm.Context(0) as ctx:
        rc = rtm.lib().rtm_eikonal(ctx.h, 1, 1, 10.0, 10.0, ns, C.c_void_p(vel.data_ptr()), nsrc,
                                   src.ctypes.data, src.ctypes.data, 1, rec.ctypes.data,
                                   rec.ctypes.data, 0, 0, C.c_void_p(out.data_ptr()), None, None, None)
        assert rc == rtm.RTM_ERR_ARG
        torch.cuda.synchronize()
        assert torch.all(out == -7.0)
        # and the context still solves
        t = torch.zeros((1, 1, 1), device="cuda")
        ctx.eikonal(vel[:1], 10.0, 10.0, [0], [0], [0], [0], times=t)
        assert t.item() == 0.0
