"""The work that a program has this library do, at the sizes of the repository's
configurations: whole sweeps (one instance, a batch, per-node trees; FP64, the
default, and the mixed precisions), the energy with its gradient, the
measurements of a finished state (FP64 energy, a density matrix), and the
allocation-free close product.

A sweep pass loads a state, advances it by one sweep and reads it back, as a
driver that checkpoints or compares runs does; the state is the seeded random
start that the repository's workloads use.  The mixed precisions' tensors and
gradients are taken in single precision, which is what their next contraction
reads.
"""
import ctypes
import math
import types

import numpy as np
import torch

from paper_1905_01331_gb300 import Sweeper, _abi
from paper_1905_01331_gb300.autograd import energy

X = np.array([[0.0, 1.0], [1.0, 0.0]])
Z = np.array([[1.0, 0.0], [0.0, -1.0]])
IY = np.array([[0.0, 1.0], [-1.0, 0.0]])


# -- models -------------------------------------------------------------------

def model_of(kind, L, h, Ly=1):
    """A periodic chain or thin torus as one-site and product terms."""
    if kind == "tfim":
        return types.SimpleNamespace(Lx=L, Ly=1, o=-h * X, A=np.stack([-Z]), B=np.stack([Z]))
    if kind == "heisenberg":
        return types.SimpleNamespace(Lx=L, Ly=1, o=np.zeros((2, 2)), A=np.stack([X, IY, Z]),
                                     B=np.stack([X, -IY, Z]))

    def on(op, n):
        out = np.ones((1, 1))
        for j in range(Ly):
            out = np.kron(out, op if j == n else np.eye(2))
        return out

    o = sum(h * on(Z, n) for n in range(Ly))
    o = o - sum(on(X, n) @ on(X, (n + 1) % Ly) for n in range(Ly))
    return types.SimpleNamespace(Lx=L, Ly=Ly, o=o, A=np.stack([-on(X, n) for n in range(Ly)]),
                                 B=np.stack([on(X, n) for n in range(Ly)]))


def problems(case):
    """[(model, L, chi)] of a case: one instance, or a batch of chains whose
    fields, lengths and bond dimensions are spread like the batched workload's."""
    if not case.get("count"):
        h = 3.04 if case["model"] == "torus" else 1.0
        return [(model_of(case["model"], case["L"], h, case.get("Ly", 1)), case["L"], case["chi"])]
    mix = np.random.default_rng(case["mix"])
    out = []
    for _ in range(case["count"]):
        L, chi = int(mix.choice([64, 128, 256, 512])), int(mix.choice([32, 64, 128]))
        out.append((model_of("tfim", L, float(mix.uniform(0.5, 1.5))), L, chi))
    return out


def bonds(L, d0, chi):
    chis = [d0]
    while len(chis) < int(math.log2(L)):
        chis.append(min(chi, chis[-1] ** 2))
    return chis


def shapes_of(L, d0, chi, per_node):
    chis = bonds(L, d0, chi)
    ws = [((L >> (t + 1)) if per_node else 1, chis[t + 1], chis[t], chis[t])
          for t in range(len(chis) - 1)]
    return ws, (chis[-1], chis[-1])


def start(L, d0, chi, per_node, seed):
    """Random isometries (QR of Gaussian matrices) and a normalised top tensor."""
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    shapes, vshape = shapes_of(L, d0, chi, per_node)
    ws = []
    for N, P, n, _ in shapes:
        q, r = torch.linalg.qr(torch.randn(N, n * n, P, generator=g, device="cuda", dtype=torch.float64))
        q = q * torch.sign(torch.diagonal(r, dim1=1, dim2=2))[:, None, :]
        ws.append(q.transpose(1, 2).contiguous().reshape((N, P, n, n) if per_node else (P, n, n)))
    v = torch.randn(vshape, generator=g, device="cuda", dtype=torch.float64)
    return ws, v / v.norm()


# -- the cases ----------------------------------------------------------------

def listed():
    return [
        # the smallest tree, every node its own isometry: an optimiser's step on a chain of 16
        # spins, where launches and host calls are all there is
        {"name": "grad_tfim_L16_chi8_nodes", "kind": "grad", "model": "tfim", "L": 16, "chi": 8,
         "per_node": True, "prec": "fp64"},
        # the same tree swept: the first configuration of the repository
        {"name": "sweep_tfim_L16_chi8_nodes", "kind": "sweep", "model": "tfim", "L": 16, "chi": 8,
         "per_node": True, "prec": "fp64"},
        # a plug-in's close product, with sizes that fill no tile
        {"name": "close_96x80x10007", "kind": "close", "P": 96, "Q": 80, "n2": 10007},
        # the critical chain at a small bond dimension, default precision
        {"name": "sweep_tfim_L1024_chi32_fp64", "kind": "sweep", "model": "tfim", "L": 1024,
         "chi": 32, "prec": "fp64"},
        # the headline chain in the default precision
        {"name": "sweep_tfim_L1024_chi128_fp64", "kind": "sweep", "model": "tfim", "L": 1024,
         "chi": 128, "prec": "fp64"},
        # energy and gradient of a thin torus (16-dimensional sites, four product terms per bond)
        {"name": "grad_torus_64x4_chi64_fp64", "kind": "grad", "model": "torus", "L": 64, "Ly": 4,
         "chi": 64, "prec": "fp64"},
        # what a run reports at its end: the FP64 energy of the tensors and a density matrix
        {"name": "measure_heisenberg_L256_chi128", "kind": "measure", "model": "heisenberg",
         "L": 256, "chi": 128, "layer": 3},
        # the headline chain, 3xTF32
        {"name": "sweep_tfim_L1024_chi128_tf32x3", "kind": "sweep", "model": "tfim", "L": 1024,
         "chi": 128, "prec": "tf32x3"},
        # the largest bond dimension: a Heisenberg chain in BF16x3
        {"name": "sweep_heisenberg_L256_chi256_bf16x3", "kind": "sweep", "model": "heisenberg",
         "L": 256, "chi": 256, "prec": "bf16x3"},
        # a thin torus in plain TF32
        {"name": "sweep_torus_64x4_chi128_tf32", "kind": "sweep", "model": "torus", "L": 64, "Ly": 4,
         "chi": 128, "prec": "tf32"},
        # a field scan: independent chains of mixed length and bond dimension in one context
        {"name": "sweep_16_chains_tf32x3", "kind": "sweep", "model": "tfim", "count": 16, "mix": 4,
         "prec": "tf32x3"},
        # energy and gradient of the torus at its full bond dimension in 3xTF32
        {"name": "grad_torus_64x4_chi128_tf32x3", "kind": "grad", "model": "torus", "L": 64, "Ly": 4,
         "chi": 128, "prec": "tf32x3"},
    ]


def draw(rng):
    kind = rng.choice(["grad", "sweep", "sweep", "measure", "close"])
    if kind == "close":
        return {"kind": "close", "P": int(2 ** rng.uniform(0, 8)), "Q": int(2 ** rng.uniform(0, 8)),
                "n2": int(2 ** rng.uniform(0, 17))}
    case = {"kind": kind, "model": rng.choice(["tfim", "tfim", "heisenberg", "torus"])}
    top = 128
    if kind != "measure":
        case["prec"] = rng.choice(["fp64", "fp64", "tf32x3", "tf32", "bf16x3", "bf16"])
        if case["prec"] == "fp64":
            top = 64
    else:
        case["layer"] = rng.randint(0, 2)
    if case["model"] == "torus":
        case["Ly"] = rng.choice([2, 3, 4, 5])
        case["L"] = 2 ** rng.randint(4, 7)
    else:
        case["L"] = 2 ** rng.randint(4, 10)
    case["chi"] = min(top, 2 ** rng.randint(3, 7))
    if kind != "measure" and case["model"] == "tfim" and case["L"] <= 64 and case["chi"] <= 32:
        case["per_node"] = rng.random() < 0.5
    elif kind == "sweep" and case["model"] == "tfim" and rng.random() < 0.3:
        return {"kind": "sweep", "model": "tfim", "prec": case["prec"], "count": rng.randint(2, 6),
                "mix": rng.randrange(1000)}
    return case


# -- preparing and running ----------------------------------------------------

def _dp(t):
    return ctypes.cast(t.data_ptr(), ctypes.POINTER(ctypes.c_double))


def prepare(case, seed):
    if case["kind"] == "close":
        g = torch.Generator(device="cuda")
        g.manual_seed(seed)
        y = torch.randn(case["P"], case["n2"], generator=g, device="cuda", dtype=torch.float64)
        w = torch.randn(case["Q"], case["n2"], generator=g, device="cuda", dtype=torch.float64)
        w = w / w.norm(dim=1, keepdim=True)
        c = torch.empty(case["P"], case["Q"], device="cuda", dtype=torch.float64)
        return {"case": case, "lib": _abi.load(), "y": y, "w": w, "c": c}
    probs = problems(case)
    per_node = bool(case.get("per_node"))
    tensors = [start(L, m.o.shape[0], chi, per_node, seed + 1000 * i)
               for i, (m, L, chi) in enumerate(probs)]
    sweeper = Sweeper([m for m, _, _ in probs], [chi for _, _, chi in probs], per_node=per_node,
                      prec=case.get("prec", "fp64"))
    state = {"case": case, "sweeper": sweeper}
    if case["kind"] == "grad":
        ws, v = tensors[0]
        state["ws"] = [w.requires_grad_(True) for w in ws]
        state["v"] = v.requires_grad_(True)
        return state
    flat = [(torch.cat([w.reshape(-1) for w in ws]), v) for ws, v in tensors]
    if case["kind"] == "measure":
        _load(sweeper, 0, *flat[0])
    else:
        state["in"] = flat
        state["out"] = [(torch.empty_like(w), torch.empty_like(v)) for w, v in flat]
    return state


def _load(s, inst, w, v):
    s._check(s.lib.ttn_set_isometries(s.h, inst, _dp(w), _dp(v)), "set_isometries")


def run(state):
    case = state["case"]
    if case["kind"] == "close":
        y, w, c = state["y"], state["w"], state["c"]
        rc = state["lib"].ttn_close_noalloc(
            ctypes.c_void_p(y.data_ptr()), ctypes.c_void_p(w.data_ptr()), y.shape[0], w.shape[0],
            y.shape[1], ctypes.c_void_p(c.data_ptr()),
            ctypes.c_void_p(torch.cuda.current_stream().cuda_stream))
        if rc != 0:
            raise RuntimeError(f"ttn_close_noalloc: {rc}")
        return c
    s = state["sweeper"]
    mixed = case.get("prec", "fp64") != "fp64"
    if case["kind"] == "grad":
        leaves = [state["v"], *state["ws"]]
        e = energy(s, 0, state["v"], state["ws"], prec=case["prec"])
        grads = torch.autograd.grad(e, leaves)
        if mixed:
            e, grads = e.float(), [g.float() for g in grads]
        return {"energy": e, "grads": list(grads)}
    if case["kind"] == "measure":
        return {"energy": s.energy(0), "rdm": s.rdm(0, case["layer"], which=1)}
    for i, (w, v) in enumerate(state["in"]):
        _load(s, i, w, v)
    e = s.sweep(1)
    for i, (w, v) in enumerate(state["out"]):
        s._check(s.lib.ttn_get_isometries(s.h, i, _dp(w), _dp(v)), "get_isometries")
    out = state["out"]
    if mixed:
        out = [(w.float(), v.float()) for w, v in out]
    return {"energies": e, "tensors": [t for pair in out for t in pair]}


# -- what a pass cannot do without ---------------------------------------------

def work(case):
    if case["kind"] == "close":
        P, Q, n2 = case["P"], case["Q"], case["n2"]
        return {"bytes": 8.0 * ((P + Q) * n2 + P * Q), "flops": 2.0 * P * Q * n2}
    flops = size = 0.0
    for m, L, chi in problems(case):
        per_node, K = bool(case.get("per_node")), m.A.shape[0]
        symmetric = case["model"] != "heisenberg"
        shapes, (c, _) = shapes_of(L, m.o.shape[0], chi, per_node)
        for t, (N, P, n, _) in enumerate(shapes):
            # one-site operator on a leg of w; product over both legs (or of a P x P matrix with w)
            u1, u2 = 2.0 * N * P * n ** 3, 2.0 * N * P * P * n * n
            size += N * P * n * n
            flops += (2 + 4 * K) * u1 + (1 + 2 * K) * u2                 # ascend
            if case["kind"] == "measure":
                flops += u1 + u2 if t >= case["layer"] else 0.0          # density matrix downwards
                continue
            flops += (1 + 2 * K) * u2 if symmetric else (2 + 4 * K) * (u1 + u2)   # environment
            if t > 0 or case["kind"] == "sweep":
                flops += (1 + 2 * K) * u2 + (2 + 6 * K) * u1             # descend
            if case["kind"] == "sweep":
                flops += 2 * u2                                          # polar factor
        size += c * c
        flops += (4 + 12 * K) * 2.0 * c ** 3
    if case["kind"] == "measure":
        n = bonds(case["L"], problems(case)[0][0].o.shape[0], case["chi"])[case["layer"]]
        return {"bytes": 8.0 * (size + n * n), "flops": flops}
    return {"bytes": 16.0 * size, "flops": flops}


# -- the same in plain 64-bit torch ---------------------------------------------

def _energy64(m, ws, v, per_node):
    """<psi|H|psi> with the one-site term shifted as the library shifts it (by
    the largest eigenvalue of the bond term), the shift restored at the end."""
    d0, K = m.o.shape[0], m.A.shape[0]
    eye = np.eye(d0)
    bond = 0.5 * (np.kron(m.o, eye) + np.kron(eye, m.o)) + sum(np.kron(a, b) for a, b in zip(m.A, m.B))
    c = float(np.linalg.eigvalsh(0.5 * (bond + bond.T))[-1])
    S = m.Lx if per_node else 1
    dev = dict(dtype=torch.float64, device=v.device)
    o = torch.tensor(m.o - c * eye, **dev).expand(S, d0, d0)
    A = torch.tensor(m.A, **dev).expand(S, K, d0, d0)
    B = torch.tensor(m.B, **dev).expand(S, K, d0, d0)
    for w in ws:
        w = w if per_node else w[None]
        N, P, n, _ = w.shape
        left = (lambda x: x[0::2]) if per_node else (lambda x: x)
        right = (lambda x: x[1::2]) if per_node else (lambda x: x)
        flat = w.reshape(N, P, n * n).transpose(1, 2)

        def close(y):
            return y.reshape(N, P, n * n) @ flat

        def on_left(x):
            return x.transpose(1, 2)[:, None] @ w

        def on_right(x):
            return w @ x[:, None]

        y = on_left(left(o)) + on_right(right(o))
        for k in range(K):
            y = y + left(A)[:, k].transpose(1, 2)[:, None] @ on_right(right(B)[:, k])
        ups = ([close(on_right(right(A)[:, k])) for k in range(K)],
               [close(on_left(left(B)[:, k])) for k in range(K)])
        o, A, B = close(y), torch.stack(ups[0], 1), torch.stack(ups[1], 1)
    i, j = 0, o.shape[0] - 1
    hv = o[i] @ v + v @ o[j].T
    for k in range(K):
        hv = hv + A[i, k] @ v @ B[j, k].T + B[i, k] @ v @ A[j, k].T
    return (v * hv).sum() + c * m.Lx


def exact(case, seed):
    if case["kind"] == "sweep":
        return None
    state = prepare(case, seed)
    if case["kind"] == "close":
        return state["y"] @ state["w"].T
    m, L, chi = problems(case)[0]
    per_node = bool(case.get("per_node"))
    if case["kind"] == "grad":
        e = _energy64(m, state["ws"], state["v"], per_node)
        return {"energy": e.detach(), "grads": list(torch.autograd.grad(e, [state["v"], *state["ws"]]))}
    ws, v = start(L, m.o.shape[0], chi, per_node, seed)
    rho = v @ v.T
    for w in reversed(ws[case["layer"]:]):
        P, n, _ = w.shape
        g = (rho @ w.reshape(P, n * n)).reshape(P, n, n)
        rho = torch.einsum("plr,pmr->lm", w, g)
    return {"energy": float(_energy64(m, ws, v, per_node)), "rdm": rho.cpu().numpy()}
