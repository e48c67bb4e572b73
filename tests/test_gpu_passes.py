"""Energy and gradient passes are captured on their second call and replayed:
every call, with new tensors and a new gradient buffer, gives the bits of a
first call in a fresh context, also with recomputed operators and after a sweep
or an autotuning in between."""
import numpy as np
import pytest

import ttn_inputs as ti

pytestmark = pytest.mark.gpu


def _pass(s, seed, L, d0, chi, per_node, prec):
    import torch
    from paper_1905_01331_gb300.autograd import energy
    ws, V = ti.initial_tensors(L, d0, chi, seed, per_node)
    tw = [torch.tensor(w, device="cuda", requires_grad=True) for w in ws]
    tv = torch.tensor(V, device="cuda", requires_grad=True)
    e = energy(s, 0, tv, tw, prec=prec)
    g = torch.autograd.grad(e, [tv, *tw])
    with torch.no_grad():
        e2 = energy(s, 0, tv, tw, prec=prec)
    return [e.item(), e2.item(), s.energy(0)] + [x.cpu().numpy() for x in g]


@pytest.mark.parametrize("model,L,chi,per_node,prec,recompute", [
    ("tfim", 16, 8, True, "fp64", False), ("tfim", 64, 64, False, "fp64", False),
    ("torus", 16, 32, False, "fp64", True), ("tfim", 64, 64, False, "tf32x3", False)])
def test_replayed_passes_equal_first_calls(model, L, chi, per_node, prec, recompute):
    from paper_1905_01331_gb300 import Sweeper
    m = ti.tfim_chain(L, 1.0) if model == "tfim" else ti.tfim_torus(L, 2, 3.0)
    kw = dict(per_node=per_node, prec=prec, recompute_ops=recompute)
    s = Sweeper(m, chi, **kw)
    for call in range(5):
        got = _pass(s, 40 + call, L, m.d0, chi, per_node, prec)
        fresh = Sweeper(m, chi, **kw)
        ref = _pass(fresh, 40 + call, L, m.d0, chi, per_node, prec)
        fresh.close()
        for a, b in zip(got, ref):
            assert np.array_equal(a, b)
        if call == 2:
            s.sweep(2)
    s.close()
