"""FP64 gradient passes whose layer products have more digit-engine tiles than
the GPU has SMs, so that they run as equal shares of 16-column blocks with the
small operand's digits ready in memory: one and two row tiles, one to three
batches, symmetric and other operator factors, against the oracle's
environments."""
import numpy as np
import pytest

import ttn_inputs as ti
from oracle import ttn as oracle

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("model,L,chi", [
    ("tfim", 64, 128), ("heisenberg", 64, 128), ("torus", 32, 128), ("tfim", 64, 256)])
def test_gradient_of_large_layers(model, L, chi):
    """The oracle adds at most n^2 < 2^16 terms per output in FP64 (2^16 2^-53 =
    7e-12 of the largest magnitude); the digit products add less."""
    import torch
    from paper_1905_01331_gb300 import Sweeper
    from paper_1905_01331_gb300.autograd import energy
    m = {"tfim": lambda: ti.tfim_chain(L, 1.0), "heisenberg": lambda: ti.heisenberg_xxx(L),
         "torus": lambda: ti.tfim_torus(L, 4, 3.0)}[model]()
    ws, V = ti.initial_tensors(L, m.d0, chi, 11)
    st = oracle.make_state(m, ws, V)
    s = Sweeper(m, chi)
    tw = [torch.tensor(w, device="cuda", requires_grad=True) for w in st.ws]
    tv = torch.tensor(st.V, device="cuda", requires_grad=True)
    E = energy(s, 0, tv, tw)
    g = torch.autograd.grad(E, tw)
    s.close()
    assert abs(E.item() - oracle.energy(st)) < 1e-11 * abs(E.item())
    for t, x in enumerate(g):
        ref = oracle.env_layer(st, t)
        assert np.abs(x.cpu().numpy() - ref).max() < 1e-11 * np.abs(ref).max(), t


def test_environments_of_a_per_node_tree():
    """Batches of nodes and parent indices: 16 nodes of 64 x 64 products, one
    operator per node; the bound as above (2^12 terms)."""
    from paper_1905_01331_gb300 import Sweeper
    m = ti.tfim_chain(256, 1.0)
    ws, V = ti.initial_tensors(256, m.d0, 64, 11, True)
    st = oracle.make_state(m, ws, V, per_node=True)
    s = Sweeper(m, 64, per_node=True)
    s.set_isometries(0, ws, V)
    for t in range(2, len(ws)):
        ref = oracle.env_layer(st, t)
        got = s.env(0, t).cpu().numpy()
        assert np.abs(got - ref).max() < 1e-11 * max(1.0, np.abs(ref).max()), t
    s.close()
