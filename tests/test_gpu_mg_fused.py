"""The fused pieces of the multigrid cycle (2D sweeps on overlapped 16 x 16 and 32 x 32 tiles, residual with
restriction, the one-CTA bottom) against the oracle's cycle: boxes whose levels end inside a tile, every smoothing
count from none to three on either side, both orders, both smoothers, 2D and 3D.

FP64 repeats the oracle's cycle up to rounding: 1e-12 of the maximum, as in test_gpu_mg.py.  FP32: one operation of a
sweep or residual errs by at most eps32 (1 + |c0|) max|x| (c0 the centre coefficient of a L_h), a cycle of up to six
sweeps a level takes fewer than 64 such operations in a row at a point."""
import math

import numpy as np
import pytest
import torch

import ew_inputs
from oracle import oracle as O

pytestmark = pytest.mark.gpu
EPS32 = float(np.finfo(np.float32).eps)


@pytest.fixture(scope="module")
def ew():
    import __graft_entry__
    __graft_entry__.build()
    import paper_2507_18282_gb300 as ew
    return ew


@pytest.mark.parametrize("prec", ["fp64", "fp32"])
@pytest.mark.parametrize("red_black", [False, True])
@pytest.mark.parametrize("order", [2, 4])
@pytest.mark.parametrize("n,pre,post", [((7, 9), 1, 1), ((63, 31), 2, 2), ((63, 127), 1, 2), ((95, 79), 3, 0),
                                        ((191, 47), 0, 3), ((127, 255), 2, 1), ((447, 383), 2, 2), ((15, 31, 7), 1, 2),
                                        ((31, 23, 15), 0, 1)])
def test_cycles_against_the_oracle(ew, prec, red_black, order, n, pre, post):
    L = tuple((m + 1) / (n[0] + 1) for m in n)
    g = ew.ew_grid_create(len(n), n, L, order=order, prec=prec)
    og = O.Grid(n, L, order)
    a = 0.5 * (2 * math.pi / (12.0 * 10)) ** 2
    b = ew_inputs.uniform_pm1(51, og.size).astype(np.float32).astype(np.float64)
    x0 = ew_inputs.uniform_pm1(52, og.size).astype(np.float32).astype(np.float64)
    dt = torch.float64 if prec == "fp64" else torch.float32
    x = torch.tensor(x0, dtype=dt, device="cuda")
    mg = ew.mg_params(pre=pre, post=post, max_cycles=2, red_black=red_black)
    ew.ew_implicit_step_mg(g, a, torch.tensor(b, dtype=dt, device="cuda"), x, mg)
    ref, _ = O.mg_solve(og, a, b, x0=x0, ncycles=2, nu1=pre, nu2=post, red_black=red_black)
    c0 = a * sum((2.0 if order == 2 else 2.5) * ((m + 1) / l) ** 2 for m, l in zip(n, L))
    tol = 1e-12 if prec == "fp64" else 64 * EPS32 * (1 + c0)
    scale = max(np.max(np.abs(ref)), np.max(np.abs(x0)))
    assert np.max(np.abs(x.double().cpu().numpy() - ref)) <= tol * scale
    g.close()
