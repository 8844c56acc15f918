"""Wave-solves of the fewest time steps, N_t = 2 upwards, on shapes whose kernels are tuned first (the candidates advance
more steps than the solve has), against the FP64 oracle.

Tolerance: |W^n| <= 2 |v| in the 2-norm (stable steps from rest), and n steps of at most 16 roundings a point put
W^n within 16 n eps 2 |v| (n <= N_t); so the sum of the N_t + 1 weighted levels lies within
32 (N_t + 1) N_t eps max|c_n| |v| of the oracle's."""
import numpy as np
import pytest
import torch

import ew_inputs
from oracle import oracle as O

pytestmark = pytest.mark.gpu
EPS = {"fp32": 2.0**-23, "fp64": 2.0**-52, "fp32x2": 2.0**-46}


@pytest.mark.parametrize("nt", [2, 3, 4, 5])
@pytest.mark.parametrize("n,order,prec", [((70, 41, 37), 2, "fp32"), ((27, 91, 33), 2, "fp32"), ((70, 41, 37), 2, "fp64"),
                                          ((65, 35, 30), 4, "fp32"), ((1601, 903), 2, "fp32"), ((1601, 903), 4, "fp32"),
                                          ((403, 391), 2, "fp64"), ((403, 391), 4, "fp32x2")])
def test_few_steps(nt, n, order, prec):
    import __graft_entry__
    __graft_entry__.build()
    import paper_2507_18282_gb300 as ew
    L = (1.0, 0.8, 0.9)[:len(n)]
    rho = (4.0 if order == 2 else 16.0 / 3.0) * sum(((m + 1) / l) ** 2 for m, l in zip(n, L))
    omega = 2.0 * np.pi * 0.5 * np.sqrt(rho) / (0.8 * nt)
    g = ew.ew_grid_create(len(n), n, L, order=order, prec=prec)
    p = ew.filter_params(omega, steps_per_period=nt)
    v = torch.tensor(ew_inputs.uniform_pm1(61, g.size), dtype=g.dtype, device="cuda")
    w = torch.full_like(v, float("nan"))
    ew.ew_filter_apply(g, p, v, w)
    info, c = ew.ew_filter_setup(g, p)
    assert info["Nt"] == nt
    x = v.double().cpu().numpy()
    ref = O.filter_explicit(O.Grid(n, L, order), O.filter_params(omega, 1, nt), x)
    err = np.linalg.norm(w.double().cpu().numpy() - ref)
    assert err <= 32 * (nt + 1) * nt * EPS[prec] * np.max(np.abs(c)) * np.linalg.norm(x)
    g.close()
