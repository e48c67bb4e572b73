"""Digit products of operands whose rows (columns) differ in scale: every row and
every column is cut under its own power of two, so that scaling them by powers of
two scales the results and changes no bit of them, as in plain FP64 sums."""
import ctypes

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def _close(Y, W):
    import torch
    from paper_1905_01331_gb300 import _abi
    lib = _abi.load()
    dY, dW = torch.from_numpy(Y).cuda(), torch.from_numpy(W).cuda()
    C = torch.full((Y.shape[0], W.shape[0]), 7.0, dtype=torch.float64, device="cuda")
    rc = lib.ttn_close_noalloc(ctypes.c_void_p(dY.data_ptr()), ctypes.c_void_p(dW.data_ptr()),
                               Y.shape[0], W.shape[0], Y.shape[1], ctypes.c_void_p(C.data_ptr()),
                               ctypes.c_void_p(torch.cuda.current_stream().cuda_stream))
    assert rc == 0
    torch.cuda.synchronize()
    return C.cpu().numpy()


# one part of K and many, tile edges, splits with and without a remainder
SIZES = [(128, 64, 16384), (129, 65, 2047), (256, 256, 129), (96, 80, 10007), (16, 16, 70001)]


@pytest.mark.parametrize("P,Q,n2", SIZES)
def test_graded_rows_scale_the_result(P, Q, n2):
    rng = np.random.default_rng(P + Q + n2)
    Y, W = rng.standard_normal((P, n2)), rng.standard_normal((Q, n2))
    r, c = rng.integers(0, 200, (P, 1)), rng.integers(0, 200, (Q, 1))
    r[0] = c[0] = 0
    Y[P // 2] = 0.0
    plain = _close(Y, W)
    graded = _close(np.ldexp(Y, -r), np.ldexp(W, -c))
    assert np.array_equal(graded, np.ldexp(plain, -(r + c.T)))
    assert np.abs(plain - Y @ W.T).max() <= n2 * 2.0 ** -53 * (np.abs(Y) @ np.abs(W).T).max()


def test_one_large_element_leaves_the_other_rows():
    rng = np.random.default_rng(1)
    Y, W = rng.standard_normal((100, 4100)), rng.standard_normal((70, 4100))
    ref = _close(Y, W)
    Y[3, 4000] = 1e10
    got = _close(Y, W)
    rest = np.arange(100) != 3
    assert np.array_equal(got[rest], ref[rest])


def test_graded_products_on_every_route():
    """Streamed, split and several groups graded each in its own way, against the
    FP64 kernel: at most 384 terms per output, 2^-53 of K max|a_m| max|b_n| for
    each of them there, and 2^-57 for the digits."""
    import torch
    from paper_1905_01331_gb300 import _abi
    lib = _abi.load()
    nbytes = lib.ttn_selftest_bytes()
    ws = torch.empty(nbytes, dtype=torch.uint8, device="cuda")
    out = np.full(24, np.nan)
    rc = lib.ttn_selftest_digits(ctypes.c_void_p(ws.data_ptr()), nbytes,
                                 out.ctypes.data_as(ctypes.POINTER(ctypes.c_double)), 24,
                                 ctypes.c_void_p(torch.cuda.current_stream().cuda_stream))
    assert rc == 0
    assert (out[1::2] == 0).all(), out
    assert (out[16::2] <= 384 * 2.0 ** -53 + 2.0 ** -57).all(), out
