"""Captured energy and gradient passes: when a pass is captured, and that a replay is
the pass that was asked for -- of its own instance, precision and table of tuned
configurations, with other passes of the same context in between."""
import ctypes

import numpy as np
import pytest

import ttn_inputs as ti

pytestmark = pytest.mark.gpu


def _grad(s, inst, seed, L, d0, chi, prec):
    import torch
    from paper_1905_01331_gb300.autograd import energy
    ws, V = ti.initial_tensors(L, d0, chi, seed)
    tw = [torch.tensor(w, device="cuda", requires_grad=True) for w in ws]
    tv = torch.tensor(V, device="cuda", requires_grad=True)
    e = energy(s, inst, tv, tw, prec=prec)
    return [e.item()] + [x.cpu().numpy() for x in torch.autograd.grad(e, [tv, *tw])]


def _same(a, b):
    return all(np.array_equal(x, y) for x, y in zip(a, b))


def test_a_few_calls_pay_for_no_capture():
    """The host enqueues a pass's launches in its first three calls and once more
    for the capture; a replay enqueues none of them."""
    import torch
    from paper_1905_01331_gb300 import Sweeper
    m = ti.tfim_chain(64, 1.0)
    s = Sweeper(m, 16)
    ws, V = ti.initial_tensors(64, 2, 16, 3)
    s.set_isometries(0, ws, V)
    E, counts, energies = ctypes.c_double(), [s.launch_count], []
    for _ in range(6):
        s._check(s.lib.ttn_energy(s.h, 0, ctypes.byref(E)), "energy")
        counts.append(s.launch_count)
        energies.append(E.value)
    s.close()
    new = np.diff(counts)
    assert new[0] > 0 and (new[:4] == new[0]).all() and (new[4:] == 0).all(), new
    assert len(set(energies)) == 1


def test_replays_of_two_instances_and_precisions():
    """Two instances of different size, FP64 and 3xTF32 passes, energies and
    gradients in turn, from a pass's first call to its second replay: each gives the
    bits of a fresh context of that one instance."""
    from paper_1905_01331_gb300 import Sweeper
    sizes = [(64, 64), (32, 32)]
    models = [ti.tfim_chain(L, 0.8 + 0.3 * i) for i, (L, _) in enumerate(sizes)]
    both = Sweeper(models, [chi for _, chi in sizes], prec="tf32x3")
    for call in range(6):
        for i, (L, chi) in enumerate(sizes):
            for prec in ("fp64", "tf32x3"):
                seed = 100 * call + 10 * i
                got = _grad(both, i, seed, L, 2, chi, prec) + [both.energy(i)]
                one = Sweeper(models[i], chi, prec="tf32x3")
                ref = _grad(one, 0, seed, L, 2, chi, prec) + [one.energy(0)]
                one.close()
                assert _same(got, ref), (call, i, prec)
    both.close()


@pytest.mark.parametrize("prec", ["fp64", "tf32x3"])
def test_autotuning_ends_the_replay_of_older_choices(prec):
    """After an autotuning, a pass that was being replayed runs with the new
    table: the bits of a fresh context created with that table, in every call."""
    from paper_1905_01331_gb300 import Sweeper
    L, chi = 128, 64
    m = ti.tfim_chain(L, 1.0)
    s = Sweeper(m, chi, prec=prec)
    for call in range(5):
        _grad(s, 0, call, L, 2, chi, prec)
    table = s.autotune(reps=2)
    for call in range(6):
        got = _grad(s, 0, 20 + call, L, 2, chi, prec)
        fresh = Sweeper(m, chi, prec=prec, tiles=table)
        ref = _grad(fresh, 0, 20 + call, L, 2, chi, prec)
        fresh.close()
        assert _same(got, ref), call
    s.close()
