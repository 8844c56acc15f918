"""The Rayleigh-Ritz step's host eigen-solver (csrc/ew_small_eig.h), compiled by itself, against the definition: A V = V w
and V^T V = I.  Sizes from one row up, clustered and repeated eigenvalues, banded, diagonal and zero matrices.

Tolerance: the backward error of the reflections and of fewer than 2 n QR steps is at most a small multiple of n eps |A|;
16 n eps |A| for the residual, 16 n eps for the orthogonality."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

CSRC = os.path.join(os.path.dirname(__file__), "..", "paper_2507_18282_gb300", "csrc")
EPS = float(np.finfo(float).eps)


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    d = tmp_path_factory.mktemp("small_eig")
    (d / "t.cpp").write_text("""
#include "ew_small_eig.h"
extern "C" void run(int n, const double* a, double* v, double* w) {
    std::vector<double> A(a, a + (size_t)n * n), V, W;
    ew::tridiagonal_eig(n, A, V, W);
    std::copy(V.begin(), V.end(), v);
    std::copy(W.begin(), W.end(), w);
}
""")
    so = str(d / "t.so")
    subprocess.run(["g++", "-O3", "-shared", "-fPIC", "-I", CSRC, "-o", so, str(d / "t.cpp")], check=True)
    return ctypes.CDLL(so)


def _matrix(kind, n):
    rng = np.random.default_rng(n)
    if kind == "zero":
        return np.zeros((n, n))
    if kind == "diagonal":
        return np.diag(rng.standard_normal(n))
    if kind == "banded":
        A = np.triu(np.tril(rng.standard_normal((n, n)), 3), -3)
        return A + A.T
    if kind == "dense":
        A = rng.standard_normal((n, n))
        return A + A.T
    Q = np.linalg.qr(rng.standard_normal((n, n)))[0]
    w = np.where(np.arange(n) < n // 2, 1.0, -0.2) if kind == "repeated" else 1.0 - 1e-9 * (np.arange(n) % 3)
    A = (Q * w) @ Q.T
    return 0.5 * (A + A.T)


@pytest.mark.parametrize("kind", ["zero", "diagonal", "banded", "dense", "repeated", "clustered"])
@pytest.mark.parametrize("n", [1, 2, 3, 5, 16, 33, 112, 150])
def test_definition(lib, kind, n):
    A = np.ascontiguousarray(_matrix(kind, n))
    V, w = np.full((n, n), np.nan), np.full(n, np.nan)
    ptr = [x.ctypes.data_as(ctypes.c_void_p) for x in (A, V, w)]
    lib.run(n, *ptr)
    norm = np.linalg.norm(A, 2)
    assert np.max(np.abs(A @ V - V * w)) <= 16 * n * EPS * norm
    assert np.max(np.abs(V.T @ V - np.eye(n))) <= 16 * n * EPS
