"""The eigenvector of the Lanczos tridiagonal from its twisted factorisation, run on
the host: it decides the convergence checks and gives the mixed modes' vector.
Tridiagonals of unit size, as the kernel scales them, with the lowest eigenvalue of
numpy; the residual |T z - th z| / |z| is the rounding of the recurrences: 48 bits
in pair arithmetic, 53 in FP64, a few operations per row."""
import os
import shutil
import subprocess

import numpy as np
import pytest

HERE = os.path.dirname(os.path.abspath(__file__))


@pytest.fixture(scope="module")
def driver(tmp_path_factory):
    gxx = shutil.which("g++")
    if gxx is None:
        pytest.skip("g++ not available")
    exe = str(tmp_path_factory.mktemp("twist") / "driver")
    subprocess.run([gxx, "-O2", "-std=c++17", "-ffp-contract=off", "-o", exe, os.path.join(HERE, "twisted_driver.cpp")],
                   check=True)
    return exe


def _cases():
    rng = np.random.default_rng(5)
    out = []
    for t in range(300):
        m = int(rng.integers(1, 50))
        a, b = rng.normal(size=m), np.abs(rng.normal(size=max(m - 1, 0))) + 0.02
        if t % 4 == 1:                 # a vector that decays towards the end (a converged cycle)
            a[m // 2:] += 20
            b[m // 2:] *= 1e-3
        if t % 4 == 2:                 # zeros on the diagonal (a shifted recurrence starts with one)
            a[rng.integers(0, m, 2)] = 0.0
        if t % 4 == 3 and m > 3:       # nearly decoupled
            b[m // 3] = 1e-9
        s = 1.0 / (max(np.abs(a).max(), np.abs(b).max() if m > 1 else 0.0) or 1.0)   # (a single zero stays)
        out.append((a * s, b * s))
    out.append((np.zeros(4), np.ones(3)))                   # zero pivots at th = 0 +- ...
    return out


def test_residual_and_last_component(driver):
    cases, ths = _cases(), []
    text = ""
    for a, b in cases:
        T = np.diag(a) + np.diag(b, 1) + np.diag(b, -1)
        w, V = np.linalg.eigh(T)
        ths.append((T, w, V))
        text += f"{len(a)} " + " ".join(f"{x:.17g}" for x in [w[0], *a, *b]) + "\n"
    lines = subprocess.run([driver], input=text, capture_output=True, text=True, check=True).stdout.strip().split("\n")
    assert len(lines) == len(cases)
    for line, (T, w, V) in zip(lines, ths):
        m = len(w)
        z = np.array([float(x) for x in line.split()])
        for vec, eps in ((z[:m], 2.0 ** -46), (z[m:], 2.0 ** -50)):
            assert np.isfinite(vec).all()
            n = np.linalg.norm(vec)
            assert np.linalg.norm(T @ vec - w[0] * vec) / n <= 8 * m * eps
            if m > 1 and w[1] - w[0] > 1e-6:
                gap = w[1] - w[0]
                assert abs(abs(vec[-1]) / n - abs(V[-1, 0])) <= 8 * m * eps / gap + 1e-13


def test_zero_pivots(driver):
    """th equal to the first diagonal entry: the first pivot is zero and replaced."""
    text = "3 0.0 0.0 0.0 0.0 1.0 1.0\n2 0.5 0.5 0.5 0.0\n1 0.25 0.25\n"
    out = subprocess.run([driver], input=text, capture_output=True, text=True, check=True).stdout.strip().split("\n")
    z = np.array([float(x) for x in out[0].split()])[:3]
    assert np.allclose(np.abs(z) / np.linalg.norm(z), np.array([1, 0, 1]) / np.sqrt(2), atol=1e-12)
    assert all(np.isfinite(float(x)) for line in out for x in line.split())
