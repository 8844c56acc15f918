"""A solution that the number format holds exactly is left as it is by the multigrid cycle, bit for bit: x of small
integers, dyadic stencil coefficients and b = M x make every term of b - M x exact, so the residual is 0 on every
point, and an update x + w (b - M x) returns x.  (An update with its constants multiplied out rounds instead, and the
lowest residual a solve can reach rises with it.)  Both tile sizes of the 2D sweeps, one to three sweeps on either
side, 3D levels, both orders and smoothers."""
import numpy as np
import pytest
import torch

from oracle import oracle as O

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec", ["fp64", "fp32"])
@pytest.mark.parametrize("red_black", [False, True])
@pytest.mark.parametrize("order", [2, 4])
@pytest.mark.parametrize("n,pre,post", [((31, 63), 2, 2), ((127, 127), 1, 3), ((127, 63), 0, 2), ((511, 511), 2, 1),
                                        ((31, 15, 31), 2, 1)])
def test_exact_solution_stays(prec, red_black, order, n, pre, post):
    import __graft_entry__
    __graft_entry__.build()
    import paper_2507_18282_gb300 as ew
    h = 1.0 / (n[0] + 1)
    L = tuple((m + 1) * h for m in n)  # the same power of two h on every axis
    a = (1.0 if order == 2 else 12.0) * h * h / 8.0  # off-centre coefficients 1/8, or 2 and -1/8
    rng = np.random.default_rng(7)
    x = rng.integers(-8, 9, size=int(np.prod(n))).astype(np.float64)
    mx = np.asarray(O.apply_M(O.Grid(n, L, order), a, x)).ravel()
    b = np.round(mx * 8.0) / 8.0  # M x, whose values are multiples of 1/8
    assert np.max(np.abs(b - mx)) < 1e-11
    g = ew.ew_grid_create(len(n), n, L, order=order, prec=prec)
    xd = torch.tensor(x, dtype=g.dtype, device="cuda")
    ew.ew_implicit_step_mg(g, a, torch.tensor(b, dtype=g.dtype, device="cuda"), xd,
                           ew.mg_params(pre=pre, post=post, max_cycles=2, red_black=red_black))
    assert np.array_equal(xd.double().cpu().numpy(), x)
    g.close()
