"""The eigen-solver's Gram products and block updates at sizes off their tiles: blocks of one to seven vectors, bases that
are no multiple of four, boxes of fewer points than a thread block and of a few rows a thread.

Tolerance: the solver's own stopping test, tol = 1e-11 on the residual of S; the eigenvalues of L then agree with the
closed form to the 1e-9 used in test_gpu_eigs.py."""
import numpy as np
import pytest

from oracle import oracle as O
from test_gpu_eigs import _solve, _wanted, ew  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,block,krylov,nw", [((9, 13), 1, 17, 3), ((37, 23), 5, 31, 6), ((61, 67), 7, 43, 5),
                                               ((131, 95), 3, 26, 5)])
def test_ragged_blocks(ew, n, block, krylov, nw):
    L, omega, Np = (1.2, 0.8), 30.0, 2
    lam, rep, info, _ = _solve(ew, n, L, 2, "fp64", omega, Np, nw, block, krylov, tol=1e-11)
    og = O.Grid(n, L, 2)
    want, _, _ = _wanted(og, O.filter_params(omega, Np, info["steps_per_period"]), nw)
    assert rep["n_converged"] == nw
    np.testing.assert_allclose(np.sort(lam), np.sort(want), rtol=1e-9)
