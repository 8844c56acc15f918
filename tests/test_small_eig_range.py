"""The Rayleigh-Ritz step's host eigen-solver on matrices whose entries' squares leave the range of doubles, and on
off-diagonals far below the diagonal's resolution: A V = V w and V^T V = I with the bounds of test_small_eig.py (16 n eps
|A| and 16 n eps), the residual relative to the matrix's scale."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

CSRC = os.path.join(os.path.dirname(__file__), "..", "paper_2507_18282_gb300", "csrc")
EPS = float(np.finfo(float).eps)


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    d = tmp_path_factory.mktemp("small_eig_range")
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


@pytest.mark.parametrize("exponent", [-1000, -660, -530, 530, 660, 1000])
@pytest.mark.parametrize("n", [2, 3, 5, 33])
def test_scaled(lib, n, exponent):
    rng = np.random.default_rng(n)
    B = rng.standard_normal((n, n))
    B = np.ascontiguousarray(B + B.T)
    B[np.diag_indices(n)] = 0.0
    A = np.ldexp(B, exponent)
    V, w = np.full((n, n), np.nan), np.full(n, np.nan)
    lib.run(n, *[x.ctypes.data_as(ctypes.c_void_p) for x in (A, V, w)])
    w = np.ldexp(w, -exponent)
    assert np.max(np.abs(B @ V - V * w)) <= 16 * n * EPS * np.linalg.norm(B, 2)
    assert np.max(np.abs(V.T @ V - np.eye(n))) <= 16 * n * EPS


@pytest.mark.parametrize("tiny", [1e-170, 1e-300])
def test_tiny_coupling_of_zeros(lib, tiny):
    A = np.diag([1.0, 0.0, 0.0])
    A[1, 2] = A[2, 1] = tiny
    V, w = np.full((3, 3), np.nan), np.full(3, np.nan)
    lib.run(3, *[x.ctypes.data_as(ctypes.c_void_p) for x in (A, V, w)])
    assert np.max(np.abs(A @ V - V * w)) <= 48 * EPS
    assert np.max(np.abs(V.T @ V - np.eye(3))) <= 48 * EPS
