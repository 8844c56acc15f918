"""The FP32 3D steps blocked over time (64 x 32 points a CTA, z cut into chunks) at the edges of their tiles: one
point, exact owned tiles (56 x 24 at depths 2 of order 4 and 4 of order 2, 56 x 26 at depth 3), one more or less, odd
and even rows, chunks of a few planes, N_t not a multiple of the depth, every face kind.

Fourth order takes the operations of the one-step kernel in their order: bit for bit equal to temporal_block = 1.
Second order differs from it in rounding only: each against the FP64 oracle within 4 N_t eps32 ||v||, the bound of the
other FP32 wave-solve tests, and equal bit for bit at depths 2, 3, 4 and the tuned one."""
import numpy as np
import pytest
import torch

import ew_inputs
from oracle import oracle as O

pytestmark = pytest.mark.gpu
EPS32 = float(np.finfo(np.float32).eps)
SIZES = [((1, 1, 1), 1), ((3, 2, 5), 2), ((56, 24, 9), 1), ((57, 23, 31), 1), ((55, 25, 30), 2), ((112, 26, 17), 1),
         ((113, 53, 64), 1), ((62, 61, 150), 3), ((170, 49, 4), 1)]


@pytest.fixture(scope="module")
def ew():
    import __graft_entry__
    __graft_entry__.build()
    import paper_2507_18282_gb300 as ew
    return ew


def _apply(ew, n, order, bc, nvec, tb, spp):
    L = (1.0, 0.9, 0.8)
    g = ew.ew_grid_create(3, n, L, order=order, prec="fp32", bc=list(bc))
    rho = (4.0 if order == 2 else 16.0 / 3.0) * sum(((m + 1) / l) ** 2 for m, l in zip(n, L))
    omega = 2.0 * np.pi * 0.5 * np.sqrt(rho) / (0.8 * spp)
    p = ew.filter_params(omega, num_periods=1, steps_per_period=spp, temporal_block=tb)
    v = torch.tensor(ew_inputs.uniform_pm1(3, g.size * nvec), dtype=torch.float32, device="cuda")
    w = torch.full_like(v, float("nan"))
    ew.ew_filter_apply(g, p, v, w, nvec=nvec)
    torch.cuda.synchronize()
    size = g.size
    g.close()
    return v, w, omega, size, L


@pytest.mark.parametrize("bc", ["DDDDDD", "NDDNDN", "NNNNNN"])
@pytest.mark.parametrize("n,nvec", SIZES)
@pytest.mark.parametrize("spp", [11, 12])
def test_order4_equals_one_step_a_launch(ew, n, nvec, bc, spp):
    a = _apply(ew, n, 4, bc, nvec, 0, spp)[1]
    assert torch.equal(a, _apply(ew, n, 4, bc, nvec, 1, spp)[1])
    assert torch.equal(a, _apply(ew, n, 4, bc, nvec, 3, spp)[1])


@pytest.mark.parametrize("bc", ["DDDDDD", "NDDNDN", "NNNNNN"])
@pytest.mark.parametrize("n,nvec", SIZES[1:])  # the oracle takes no axis of one interior point with Neumann faces
def test_order2_depths(ew, n, nvec, bc):
    spp = 12
    v, a, omega, size, L = _apply(ew, n, 2, bc, nvec, 0, spp)
    for tb in (2, 3, 4):
        assert torch.equal(a, _apply(ew, n, 2, bc, nvec, tb, spp)[1])
    og, prm = O.Grid(n, L, 2, list(bc)), O.filter_params(omega, 1, spp)
    x = v[(nvec - 1) * size:].double().cpu().numpy()
    y = a[(nvec - 1) * size:].double().cpu().numpy()
    assert np.linalg.norm(y - O.filter_explicit(og, prm, x)) <= 4 * spp * EPS32 * np.linalg.norm(x)
