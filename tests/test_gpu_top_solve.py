"""The top solve's energy against the lowest eigenvalue of the same top
Hamiltonian (built from the ascended operators, its symmetric part: the mixed
modes' products leave them asymmetric by 1e-7) by ARPACK, over the top
dimensions where the kernel's staging differs: below a tile (4), one tile and
one CTA (8), grids with and without a CTA for the convergence checks, the
largest (256), and with several streams sharing the GPU."""
import numpy as np
import pytest
import scipy.sparse.linalg as spla

import ttn_inputs as ti

pytestmark = pytest.mark.gpu


def _lowest(ops, K, c):
    o, A, B = ops[0], ops[1:1 + K], ops[1 + K:]

    def mv(x):
        x = x.reshape(c, c)
        y = (o + o.T) @ x + x @ (o + o.T)
        for a, b in zip(A, B):
            y = y + a @ x @ b.T + b @ x @ a.T + a.T @ x @ b + b.T @ x @ a
        return 0.5 * y.ravel()

    if c * c <= 64:
        return np.linalg.eigvalsh(np.stack([mv(e) for e in np.eye(c * c)], 1))[0]
    op = spla.LinearOperator((c * c, c * c), matvec=mv, dtype=np.float64)
    return spla.eigsh(op, k=1, which="SA", tol=1e-12, ncv=60, return_eigenvectors=False)[0]


# residual tolerance 1e-13 |E| in FP64, 1e-8 |E| in the mixed modes: an
# eigenvalue is at most the residual away (plus the FP64 sums around it); the
# mixed modes' products of the solve carry 48 bits
@pytest.mark.parametrize("prec,tol", [("fp64", 1e-11), ("tf32x3", 2e-8)])
@pytest.mark.parametrize("chi,L", [(4, 8), (8, 16), (16, 16), (32, 32), (64, 32), (128, 64), (256, 64)])
def test_top_energy(chi, L, prec, tol):
    from paper_1905_01331_gb300 import Sweeper
    m = ti.tfim_chain(L, 1.3)
    ws, V = ti.initial_tensors(L, 2, chi, 21)
    s = Sweeper(m, chi, prec=prec, shift=0.0, lanczos_restarts=40)
    s.set_isometries(0, ws, V)
    c = s.chis()[-1]
    ref = _lowest(s.ascend(0, len(ws))[0], 1, c)
    E = s.sweep(1)[0, 0]
    assert s.top_converged
    assert abs(E - ref) <= tol * abs(ref)
    s.close()


def test_top_energy_streams():
    """Eight instances on eight streams: grids of an eighth of the GPU."""
    from paper_1905_01331_gb300 import Sweeper
    chis = [8, 16, 32, 64, 128, 128, 64, 32]
    models = [ti.tfim_chain(64, 0.9 + 0.1 * i) for i in range(8)]
    s = Sweeper(models, chis, shift=0.0, lanczos_restarts=40)
    refs = []
    for i, (m, chi) in enumerate(zip(models, chis)):
        ws, V = ti.initial_tensors(64, 2, chi, 31 + i)
        s.set_isometries(i, ws, V)
        refs.append(_lowest(s.ascend(i, len(ws))[0], 1, s.chis(i)[-1]))
    E = s.sweep(1)[0]
    assert np.abs(E - refs).max() <= 1e-11 * np.abs(refs).max()
    s.close()


@pytest.mark.parametrize("chi,L", [(2, 4), (4, 8), (8, 16)])
def test_top_energy_one_tile(chi, L):
    """One CTA with everything in shared memory (FP64, c <= 8): three product
    terms, antisymmetric factors, and a top site of its own on either side."""
    from paper_1905_01331_gb300 import Sweeper
    m = ti.heisenberg_xxx(L)
    ws, V = ti.initial_tensors(L, 2, chi, 22, True)
    s = Sweeper(m, chi, per_node=True, shift=0.0, lanczos_restarts=40)
    s.set_isometries(0, ws, V)
    c = s.chis()[-1]
    l, r = s.ascend(0, len(ws))[:2]
    H = np.kron(l[0], np.eye(c)) + np.kron(np.eye(c), r[0])
    for k in range(3):
        H = H + np.kron(l[1 + k], r[4 + k]) + np.kron(l[4 + k], r[1 + k])
    ref = np.linalg.eigvalsh(0.5 * (H + H.T))[0]
    E = s.sweep(1)[0, 0]
    assert s.top_converged
    assert abs(E - ref) <= 1e-11 * abs(ref)
    s.close()
