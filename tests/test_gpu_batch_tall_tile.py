"""Batched second-order FP32 wave-solves: the tuner times the 128 x 128 shared-memory tile at depth 16 (98 x 98 owned
points) beside the register tiles, and that tile gives the single-grid kernels' bits."""
import pytest
import torch

import ew_inputs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("bc", ["DDDD", "NDDN"])
def test_candidate_and_bits(monkeypatch, capfd, bc):
    import __graft_entry__
    __graft_entry__.build()
    import paper_2507_18282_gb300 as ew
    boxes = [(196, 98), (197, 99), (95, 301), (258, 253), (7, 1201)]
    grids, params, vin, vout = [], [], [], []
    for q, n in enumerate(boxes):
        grids.append(ew.ew_grid_create(2, n, (1.0, n[1] / n[0]), order=2, prec="fp32", bc=list(bc)))
        params.append(ew.filter_params(n[0] / (2.5 + q)))
        vin.append(torch.tensor(ew_inputs.uniform_pm1(300 + q, grids[-1].size), dtype=torch.float32, device="cuda"))
        vout.append(torch.full_like(vin[-1], float("nan")))
    monkeypatch.setenv("EW_TUNE_LOG", "1")
    ew.ew_filter_apply_batched(grids, params, vin, vout)
    torch.cuda.synchronize()
    log = capfd.readouterr().err
    line = [l for l in log.splitlines() if "batched 5 problems" in l and "tile 98x98" in l]
    assert len(line) == 1, log
    monkeypatch.setenv("EW_BATCH_VARIANT", line[0].split("variant ")[1].split()[0])
    ew.ew_filter_apply_batched(grids, params, vin, vout)
    monkeypatch.delenv("EW_TUNE_LOG")
    for q, g in enumerate(grids):
        out = torch.empty_like(vin[q])
        params[q].temporal_block = 2  # the blocked kernels, also for boxes that one CTA holds
        ew.ew_filter_apply(g, params[q], vin[q], out)
        torch.cuda.synchronize()
        assert torch.equal(out, vout[q]), boxes[q]
        g.close()
