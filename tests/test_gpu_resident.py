"""The on-chip wave-solve of small 2D grids (one CTA or a cluster of CTAs a vector) at the edges of its splits: three
rows a CTA, one row more or less, every cluster size, every number of points a thread, each face kind.

Grids that the blocked kernels serve in other calls take those kernels' operations in their order: bit for bit equal
to a call with a fixed temporal depth.  The grids of the one-CTA form are held against the FP64 oracle with the bounds
of the other wave-solve tests (FP64 1e-12 of the maximum; FP32 4 N_t eps32 |v|, pairs the same with 2^-46)."""
import numpy as np
import pytest
import torch

import ew_inputs
from oracle import oracle as O

pytestmark = pytest.mark.gpu
EPS32 = float(np.finfo(np.float32).eps)
FACES = ["DDDD", "NDDN", "DNND", "NNNN"]


@pytest.fixture(scope="module")
def ew():
    import __graft_entry__
    __graft_entry__.build()
    import paper_2507_18282_gb300 as ew
    return ew


def _apply(ew, n, order, prec, bc, nvec, tb, spp=23, seed=5):
    g = ew.ew_grid_create(2, n, (1.0, 0.8), order=order, prec=prec, bc=list(bc))
    p = ew.filter_params(_omega(n, order, spp), num_periods=1, steps_per_period=spp, temporal_block=tb)
    v = torch.tensor(ew_inputs.uniform_pm1(seed, g.size * nvec), dtype=g.dtype, device="cuda")
    w = torch.full_like(v, float("nan"))
    ew.ew_filter_apply(g, p, v, w, nvec=nvec)
    torch.cuda.synchronize()
    g.close()
    return v, w


def _omega(n, order, spp):
    rho = (4.0 if order == 2 else 16.0 / 3.0) * ((n[0] + 1) ** 2 + ((n[1] + 1) / 0.8) ** 2)
    return 2.0 * np.pi * 0.5 * np.sqrt(rho) / (0.8 * spp)


@pytest.mark.parametrize("bc", FACES)
@pytest.mark.parametrize("order", [2, 4])
@pytest.mark.parametrize("prec,n,nvec", [
    ("fp32", (1361, 48), 1),    # 16 CTAs of three rows, four points a thread
    ("fp32", (340, 193), 4),    # 13 and 12 rows, the largest grid of four vectors
    ("fp32", (129, 128), 13),   # just past the one-CTA grids, two points a thread
    ("fp64", (90, 91), 1),      # one point a thread
    ("fp64", (127, 129), 4),
    ("fp64", (103, 159), 16),
    ("fp32x2", (117, 70), 1),
    ("fp32x2", (255, 257), 3),
])
def test_cluster_equals_blocked(ew, prec, n, nvec, order, bc):
    _, a = _apply(ew, n, order, prec, bc, nvec, 0)
    _, b = _apply(ew, n, order, prec, bc, nvec, 2)
    assert torch.equal(a, b)


@pytest.mark.parametrize("bc", FACES)
@pytest.mark.parametrize("order", [2, 4])
@pytest.mark.parametrize("prec", ["fp32", "fp64", "fp32x2"])
@pytest.mark.parametrize("n,nvec", [((4, 48), 1), ((5, 49), 1), ((63, 63), 2), ((64, 47), 1), ((31, 12), 20),
                                    ((30, 31), 40), ((45, 7), 80), ((110, 80), 100)])
def test_small_grids_against_the_oracle(ew, prec, n, nvec, order, bc):
    v, w = _apply(ew, n, order, prec, bc, nvec, 0)
    size = v.numel() // nvec
    prm = O.filter_params(_omega(n, order, 23), 1, 23)
    og = O.Grid(n, (1.0, 0.8), order, list(bc))
    for j in {0, nvec - 1}:
        x = v[j * size:(j + 1) * size].double().cpu().numpy()
        y = w[j * size:(j + 1) * size].double().cpu().numpy()
        ref = O.filter_explicit(og, prm, x)
        if prec == "fp64":
            assert np.max(np.abs(y - ref)) <= 1e-12 * np.max(np.abs(ref))
        else:
            eps = EPS32 if prec == "fp32" else 2.0 ** -46
            assert np.linalg.norm(y - ref) <= 4 * 23 * eps * np.linalg.norm(x)
