"""FP64 products that also write an FP32 copy of their result: the polar factor's
first try in the mixed modes reads that copy in its correction."""
import ctypes

import numpy as np
import pytest

import ttn_inputs as ti

pytestmark = pytest.mark.gpu


def test_copy_on_every_route():
    """Digit products as tiles, streamed and split over K, and the FP64 kernel
    after a refusal.  The copy is the result rounded to FP32, entry by entry;
    the results agree to the rounding of 256 terms of at most 1 (256 2^-53 on
    sums whose largest is above 10, and as much again for the digits)."""
    import torch
    from paper_1905_01331_gb300 import _abi
    lib = _abi.load()
    nbytes = lib.ttn_selftest_bytes()
    ws = torch.empty(nbytes, dtype=torch.uint8, device="cuda")
    out = np.full(16, np.nan)
    rc = lib.ttn_selftest_digits(ctypes.c_void_p(ws.data_ptr()), nbytes,
                                 out.ctypes.data_as(ctypes.POINTER(ctypes.c_double)), 16,
                                 ctypes.c_void_p(torch.cuda.current_stream().cuda_stream))
    assert rc == 0
    assert (out[1::2] == 0).all(), out
    assert (out[::2] <= 256 * 2.0 ** -53).all(), out


@pytest.mark.parametrize("prec", ["tf32x3", "bf16x3"])
def test_factor_of_a_short_wide_layer(prec):
    """A chain of 32 spins at chi = 256: the layer with n = 16, P = 256, whose
    products over X (256 x 256 by 256 x 256) are split over K.  The isometries of
    every sweep are isometric to 1e-12 (a factor corrected with anything else
    than its own head is not)."""
    from paper_1905_01331_gb300 import Sweeper
    m = ti.tfim_chain(32, 1.0)
    ws, V = ti.initial_tensors(32, m.d0, 256, 5)
    s = Sweeper(m, 256, prec=prec)
    s.set_isometries(0, ws, V)
    for _ in range(6):
        s.sweep(1)
        got = s.get_isometries(0)[0]
        for t, w in enumerate(got):
            w = np.asarray(w).reshape(w.shape[0], -1)
            assert np.abs(w @ w.T - np.eye(w.shape[0])).max() < 1e-12, t
        print(prec, s.diagnostics(0))
    s.close()
