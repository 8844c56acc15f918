"""FP32 multigrid sweeps and residuals on 3D levels (paired columns, 64 x 32 staged regions) against the oracle's cycle:
boxes one under, at and one over the regions' 60 x 28 and 60 x 30 outputs, few planes and many.

Tolerance as in test_gpu_mg_fused.py: an operation errs by at most eps32 (1 + |c0|) max|x|, and a cycle of these sweeps
takes fewer than 64 such operations in a row at a point."""
import math

import numpy as np
import pytest
import torch

import ew_inputs
from oracle import oracle as O

pytestmark = pytest.mark.gpu
EPS32 = float(np.finfo(np.float32).eps)


@pytest.mark.parametrize("red_black", [False, True])
@pytest.mark.parametrize("order", [2, 4])
@pytest.mark.parametrize("n", [(59, 27, 7), (63, 31, 15), (119, 55, 15), (127, 63, 31), (7, 15, 127)])
def test_fp32_cycle_3d(red_black, order, n):
    import __graft_entry__
    __graft_entry__.build()
    import paper_2507_18282_gb300 as ew
    L = tuple((m + 1) / (n[0] + 1) for m in n)
    g = ew.ew_grid_create(3, n, L, order=order, prec="fp32")
    og = O.Grid(n, L, order)
    a = 0.5 * (2 * math.pi / (12.0 * 10)) ** 2
    b = ew_inputs.uniform_pm1(61, og.size).astype(np.float32).astype(np.float64)
    x0 = ew_inputs.uniform_pm1(62, og.size).astype(np.float32).astype(np.float64)
    x = torch.tensor(x0, dtype=torch.float32, device="cuda")
    mg = ew.mg_params(pre=2, post=1, max_cycles=1, red_black=red_black)
    ew.ew_implicit_step_mg(g, a, torch.tensor(b, dtype=torch.float32, device="cuda"), x, mg)
    ref, _ = O.mg_solve(og, a, b, x0=x0, ncycles=1, nu1=2, nu2=1, red_black=red_black)
    c0 = a * sum((2.0 if order == 2 else 2.5) * ((m + 1) / l) ** 2 for m, l in zip(n, L))
    scale = max(np.max(np.abs(ref)), np.max(np.abs(x0)))
    assert np.max(np.abs(x.double().cpu().numpy() - ref)) <= 64 * EPS32 * (1 + c0) * scale
    g.close()
