"""Digit products whose bounded waits run out: every wait of the kernels ends, the
context stays usable, and the caller learns of it -- by the error flag, or where
the entry point has none by NaN in every output that was not computed."""
import ctypes

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def test_expired_waits_are_not_silent():
    import torch
    from paper_1905_01331_gb300 import _abi
    lib = _abi.load()
    nbytes = lib.ttn_selftest_bytes()
    ws = torch.empty(nbytes, dtype=torch.uint8, device="cuda")
    for _ in range(2):       # (the second call: products that wait are right again)
        out = np.full(30, np.nan)
        rc = lib.ttn_selftest_digits(ctypes.c_void_p(ws.data_ptr()), nbytes,
                                     out.ctypes.data_as(ctypes.POINTER(ctypes.c_double)), 30,
                                     ctypes.c_void_p(torch.cuda.current_stream().cuda_stream))
        assert rc == 0
        assert (out[24::2] == 0).all(), out     # no output is a number
        assert (out[25::2] == 1).all(), out     # the flag is raised
        assert (out[1:24:2] == 0).all() and np.isfinite(out).all()
