"""Batched FP32 wave-solves with a tile's time levels in registers (128 columns by rows of warps): every tile shape and
depth against the single-grid kernels, bit for bit.  Boxes one point under, at and over whole tiles (104 x 84 and 96 x
76 owned points), thinner than a halo, with steps that are no multiple of the depth, Dirichlet and Neumann faces."""
import pytest
import torch

import ew_inputs

pytestmark = pytest.mark.gpu

BOXES = [((208, 168), "DDDD"), ((209, 167), "NDDN"), ((96, 380), "DDDD"), ((9, 5001), "DDDD"), ((4100, 11), "DNND"),
         ((313, 253), "NNNN"), ((511, 127), "DDDD")]


@pytest.mark.parametrize("variant", [0, 1, 2, 3])
@pytest.mark.parametrize("faces", [False, True])
def test_bits(variant, faces, monkeypatch):
    import __graft_entry__
    __graft_entry__.build()
    import paper_2507_18282_gb300 as ew
    boxes = [(n, bc if faces else "DDDD") for n, bc in BOXES]
    grids, params, vin, vout = [], [], [], []
    for q, (n, bc) in enumerate(boxes):
        L = (1.0, n[1] / n[0])
        grids.append(ew.ew_grid_create(2, n, L, order=2, prec="fp32", bc=list(bc)))
        params.append(ew.filter_params(n[0] / (3.0 + q)))
        vin.append(torch.tensor(ew_inputs.uniform_pm1(200 + q, grids[-1].size), dtype=torch.float32, device="cuda"))
        vout.append(torch.full_like(vin[-1], float("nan")))
    monkeypatch.setenv("EW_BATCH_VARIANT", str(variant))
    ew.ew_filter_apply_batched(grids, params, vin, vout)
    torch.cuda.synchronize()
    for q, g in enumerate(grids):
        out = torch.empty_like(vin[q])
        ew.ew_filter_apply(g, params[q], vin[q], out)
        torch.cuda.synchronize()
        assert torch.equal(out, vout[q]), boxes[q]
    for g in grids:
        g.close()
