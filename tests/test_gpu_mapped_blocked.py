"""The temporally blocked FP32 steps on curvilinear grids at the edges of their tiles (52 and 56 points owned of 64,
column pairs, row pitch padded to four points): exact tiles, one point more or less, odd and tiny axes, N_t not a
multiple of the depth, and blocks of vectors large enough that a CTA keeps the couplings for several.

Against the FP64 oracle with the bound of the other FP32 wave-solve tests, ||dS v|| <= 4 N_t eps32 ||v||; a vector of
a block equals its own call bit for bit (both depths take the same operations)."""
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


def _setup(ew, n, steps):
    xy = ew_inputs.mapped_vertices(n[0], n[1], "square_warp", eps=0.08)
    g = ew.ew_grid_create_mapped(n, xy, prec="fp32")
    info, _ = ew.ew_filter_setup(g, ew.filter_params(1.0, num_periods=1))
    omega = info["steps_per_period"] / (steps - 0.5)  # steps per period fall with omega
    p = ew.filter_params(omega, num_periods=1)
    info, _ = ew.ew_filter_setup(g, p)
    return g, p, omega, info, O.MappedGrid(n, xy)


@pytest.mark.parametrize("n,nvec", [((1, 1), 1), ((2, 3), 2), ((3, 70), 1), ((52, 52), 1), ((53, 51), 3),
                                    ((104, 105), 1), ((155, 157), 2), ((259, 61), 1), ((64, 208), 1)])
@pytest.mark.parametrize("steps", [8, 17])
def test_against_the_oracle(ew, n, nvec, steps):
    g, p, omega, info, m = _setup(ew, n, steps)
    v = torch.tensor(ew_inputs.uniform_pm1(9, g.size * nvec), dtype=torch.float32, device="cuda")
    w = torch.full_like(v, float("nan"))
    ew.ew_filter_apply(g, p, v, w, nvec=nvec)
    torch.cuda.synchronize()
    prm = O.filter_params(omega, 1, info["steps_per_period"])
    for j in range(nvec):
        x = v[j * g.size:(j + 1) * g.size].double().cpu().numpy()
        y = w[j * g.size:(j + 1) * g.size].double().cpu().numpy()
        assert np.linalg.norm(y - O.mapped_filter_explicit(m, prm, x)) <= 4 * info["Nt"] * EPS32 * np.linalg.norm(x)
    g.close()


@pytest.mark.parametrize("n,nvec", [((113, 57), 500), ((209, 210), 170)])
def test_block_equals_single_vectors(ew, n, nvec):
    g, p, _, _, _ = _setup(ew, n, 19)
    v = torch.tensor(ew_inputs.uniform_pm1(11, g.size * nvec), dtype=torch.float32, device="cuda")
    w, one = torch.full_like(v, float("nan")), torch.empty(g.size, dtype=torch.float32, device="cuda")
    ew.ew_filter_apply(g, p, v, w, nvec=nvec)
    for j in (0, 1, 2, nvec // 2, nvec - 1):
        ew.ew_filter_apply(g, p, v[j * g.size:(j + 1) * g.size], one, nvec=1)
        assert torch.equal(w[j * g.size:(j + 1) * g.size], one)
    assert bool(torch.isfinite(w).all())
    g.close()
