"""FP64 fourth-order Jacobi smoothing on a 2D level of more than two million points (one sweep a launch there, two
below) against the oracle's cycle: 1e-12 of the maximum, as in test_gpu_mg.py."""
import math

import numpy as np
import pytest
import torch

import ew_inputs
from oracle import oracle as O

pytestmark = pytest.mark.gpu


def test_cycle_against_the_oracle():
    import __graft_entry__
    __graft_entry__.build()
    import paper_2507_18282_gb300 as ew
    n = (2047, 1087)
    L = tuple((m + 1) / (n[0] + 1) for m in n)
    g = ew.ew_grid_create(2, n, L, order=4, prec="fp64")
    og = O.Grid(n, L, 4)
    a = 0.5 * (2 * math.pi / 120.0) ** 2
    b, x0 = ew_inputs.uniform_pm1(53, og.size), ew_inputs.uniform_pm1(54, og.size)
    x = torch.tensor(x0, device="cuda")
    ew.ew_implicit_step_mg(g, a, torch.tensor(b, device="cuda"), x, ew.mg_params(pre=2, post=1, max_cycles=1))
    ref, _ = O.mg_solve(og, a, b, x0=x0, ncycles=1, nu1=2, nu2=1)
    assert np.max(np.abs(x.cpu().numpy() - ref)) <= 1e-12 * max(np.max(np.abs(ref)), np.max(np.abs(x0)))
    g.close()
