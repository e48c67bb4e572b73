"""Products whose K splits one CTA sums itself (two accumulators in tensor
memory): the one-leg products of chi = 128 layers, whose 128 output tiles fill
most of the GPU, and those of smaller layers that still split over CTAs.  The
ascended operators against the FP64 ones."""
import numpy as np
import pytest

import ttn_inputs as ti

pytestmark = pytest.mark.gpu


# Relative Frobenius error of a chain of three full layers: a TF32 operand is
# rounded at 2^-11 (two operands, two products per layer: below 8 * 2^-11), the
# three-product form leaves FP32 accumulation, 2^-24 sqrt(16384) per product.
@pytest.mark.parametrize("prec,tol", [("tf32", 8 * 2.0 ** -11), ("tf32x3", 16 * 2.0 ** -17)])
@pytest.mark.parametrize("model,chi", [("tfim", 128), ("heisenberg", 128), ("tfim", 64)])
def test_ascended_operators(model, chi, prec, tol):
    from paper_1905_01331_gb300 import Sweeper
    m = ti.tfim_chain(64, 1.0) if model == "tfim" else ti.heisenberg_xxx(64)
    ws, V = ti.initial_tensors(64, 2, chi, 11)
    s = Sweeper(m, chi, prec=prec)
    s.set_isometries(0, ws, V)
    T = len(ws)
    got, ref = s.ascend(0, T)[0], s.ascend(0, T, prec="fp64")[0]
    for g, r in zip(got, ref):
        assert np.linalg.norm(g - r) <= tol * np.linalg.norm(r)
    s.close()
