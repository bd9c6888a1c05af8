"""The host solves that advance several chains side by side (dense.cpp, no GPU): any number of columns gives
the bits that each has alone, and a few columns cost less than a full block."""
import ctypes
import os
import subprocess
import time

import numpy as np
import pytest

from test_host_dense import CSRC, OUT, P, ROOT, lib, rand_herm  # noqa: F401 (lib is a fixture)


def _best(f, n=9):
    t = []
    for _ in range(n):
        t0 = time.perf_counter()
        f()
        t.append(time.perf_counter() - t0)
    return min(t)


def _system(n, k):
    rng = np.random.default_rng(n)
    H = rand_herm(rng, n) + 4 * np.sqrt(n) * np.eye(n)
    B = rng.standard_normal((k, n)) + 1j * rng.standard_normal((k, n))
    return H, B


def _solve(lib, H, B):  # noqa: F811
    """Columns of H X = B, one per row of the result."""
    h, x = H.copy(), B.copy()  # held while the library works on them
    assert lib.shim_cholesky_solve(len(h), P(h), P(x), len(x))
    return x


@pytest.mark.parametrize("n", [1, 2, 37, 96])
@pytest.mark.parametrize("k", [1, 2, 3, 4, 5, 8, 11, 16])
def test_cholesky_columns_alone_and_together(lib, n, k):  # noqa: F811
    H, B = _system(n, k)
    X = _solve(lib, H, B)
    for c in range(k):
        assert np.array_equal(X[c], _solve(lib, H, B[c:c + 1])[0])
    assert np.abs(X @ H.T - B).max() < 1e-12 * n


def test_few_cholesky_columns_cost_less():
    """One column took as long as eight (now a sixth), two likewise (now a quarter)."""
    so = os.path.join(OUT, "libdense_widths_shim.so")
    srcs = [os.path.join(ROOT, "tests", "shim", "dense_widths_shim.cpp"), os.path.join(CSRC, "dense.cpp")]
    os.makedirs(OUT, exist_ok=True)
    subprocess.run(["g++", "-O2", "-std=c++17", "-fPIC", "-shared", "-I", CSRC, "-o", so, *srcs], check=True)
    solve = ctypes.CDLL(so).shim_chol_solve
    solve.argtypes = [ctypes.c_int, ctypes.c_void_p, ctypes.c_void_p, ctypes.c_int]
    n = 240
    H, B = _system(n, 8)
    L = np.ascontiguousarray(np.linalg.cholesky(H))
    t = {}
    for k in (1, 2, 8):
        X = B[:k].copy()
        t[k] = _best(lambda: solve(n, P(L), P(X), k), 60)
    assert t[1] < 0.5 * t[8] and t[2] < 0.6 * t[8], t


def _tridiag(lib, d, e, lo, hi):  # noqa: F811
    w, Z = np.zeros(hi - lo), np.zeros((hi - lo, len(d)))
    lib.shim_tridiag_eig(len(d), P(d), P(e), lo, hi, P(w), P(Z))
    return w


@pytest.mark.parametrize("n", [3, 24, 100])
def test_eigenvalues_alone_and_together(lib, n):  # noqa: F811
    rng = np.random.default_rng(n)
    d, e = rng.standard_normal(n), rng.standard_normal(n)
    ref = np.linalg.eigvalsh(np.diag(d) + np.diag(e[:-1], 1) + np.diag(e[:-1], -1))
    alone = np.concatenate([_tridiag(lib, d, e, i, i + 1) for i in range(n)])
    assert np.abs(alone - ref).max() < 1e-13 * n
    for k in (1, 2, 3, 4, 5, 8, 9, 13):
        for lo in (0, n // 2):
            hi = min(n, lo + k)
            assert np.array_equal(_tridiag(lib, d, e, lo, hi), alone[lo:hi])


def test_few_eigenvalues_cost_less(lib):  # noqa: F811
    """One or two eigenpairs of a tridiagonal took almost as long as eight."""
    rng = np.random.default_rng(3)
    d, e = rng.standard_normal(100), rng.standard_normal(100)
    t = {k: _best(lambda: _tridiag(lib, d, e, 0, k), 200) for k in (1, 2, 8)}
    assert t[1] < 0.42 * t[8] and t[2] < 0.5 * t[8], t  # 0.58 and 0.63 where all took a block of eight
