"""The FP64 products on the tensor cores (eight signed base-256 digits per
operand, exact accumulation) through the entry point that takes any sizes, the
allocation-free close product C = Y W^T, against extended precision."""
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


# tile edges (128 x 64 and 128 x 32), one chunk of 128 K values and its
# remainders, odd lengths (rows that are not 16-byte aligned), the largest P, Q
SIZES = [(128, 64, 16384), (129, 65, 2047), (127, 33, 2049), (16, 16, 65536), (17, 31, 40007),
         (256, 256, 129), (256, 255, 128), (256, 256, 127), (256, 200, 8200), (96, 80, 10007)]


@pytest.mark.parametrize("P,Q,n2", SIZES)
@pytest.mark.parametrize("spread", [0, 40])
def test_close_product_error_bound(P, Q, n2, spread):
    """Worst case of the digit products: the cut of both operands (2^-61 of the
    largest magnitude each) and the dropped digit pairs (7 * 2^-62 of the powers
    of two above the two largest magnitudes) stay below 2^-57 max|Y| max|W| per
    term; each of at most 80 partial sums is rounded once and added once."""
    rng = np.random.default_rng(P * 1000 + Q + n2)
    Y = rng.standard_normal((P, n2)) * np.exp2(-rng.integers(0, spread + 1, (P, n2)))
    W = rng.standard_normal((Q, n2)) * np.exp2(-rng.integers(0, spread + 1, (Q, n2)))
    W *= 1e-5
    rows = rng.integers(0, P, 12)
    got = _close(Y, W)
    ref = Y[rows].astype(np.longdouble) @ W.T.astype(np.longdouble)
    bound = (80 * 2.0 ** -53 * (np.abs(Y[rows]) @ np.abs(W).T)
             + n2 * 2.0 ** -57 * np.abs(Y).max() * np.abs(W).max())
    assert (np.abs(got[rows] - ref) <= bound).all()


def test_close_product_special_values():
    """Infinities, NaN and zero operands give what plain FP64 sums give, and
    operands far from 1 keep their accuracy."""
    rng = np.random.default_rng(3)
    Y, W = rng.standard_normal((130, 4097)), rng.standard_normal((70, 4097))
    ref = Y @ W.T
    tol = 1e-12 * np.abs(ref).max()
    for sy, sw in ((2.0 ** 400, 2.0 ** -390), (2.0 ** -500, 2.0 ** 470), (2.0 ** -1000, 2.0 ** 900)):
        assert np.abs(_close(Y * sy, W * sw) / (sy * sw) - ref).max() <= tol
    assert (_close(0 * Y, W) == 0).all()
    Yi = Y.copy()
    Yi[3, 5], Yi[7, 6], Yi[100, 4096] = np.inf, np.nan, -np.inf
    with np.errstate(invalid="ignore"):
        refi = Yi @ W.T
    got = _close(Yi, W)
    assert np.array_equal(np.isnan(got), np.isnan(refi))
    assert np.array_equal(np.isposinf(got), np.isposinf(refi))
    assert np.array_equal(np.isneginf(got), np.isneginf(refi))
    fin = np.isfinite(refi)
    assert np.abs(got[fin] - refi[fin]).max() <= tol
