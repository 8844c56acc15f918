"""The one-launch wave-solve of 2D FP32 boxes that fit on the chip (tiles exchanging halos through tagged records)
against the blocked kernels at a fixed depth: the same operations per point, so bit for bit equal.  Sizes around the
tile splits of every region shape, uneven shares, one tile in an axis, each face kind, several vectors, N_t - 1 a
multiple of the exchange depth or not; and an exchange that never completes, which must end in EW_ETIMEOUT."""
import numpy as np
import pytest
import torch

import ew_inputs

pytestmark = pytest.mark.gpu
FACES = ["DDDD", "NDDN", "NNNN"]


@pytest.fixture(scope="module")
def ew():
    import __graft_entry__
    __graft_entry__.build()
    import paper_2507_18282_gb300 as ew
    return ew


def _apply(ew, n, order, bc, nvec, tb, spp):
    g = ew.ew_grid_create(2, n, (1.0, 0.8), order=order, prec="fp32", bc=list(bc))
    rho = (4.0 if order == 2 else 16.0 / 3.0) * ((n[0] + 1) ** 2 + ((n[1] + 1) / 0.8) ** 2)
    p = ew.filter_params(2.0 * np.pi * 0.5 * np.sqrt(rho) / (0.8 * spp), steps_per_period=spp, temporal_block=tb)
    v = torch.tensor(ew_inputs.uniform_pm1(13, g.size * nvec), dtype=torch.float32, device="cuda")
    w = torch.full_like(v, float("nan"))
    ew.ew_filter_apply(g, p, v, w, nvec=nvec)
    torch.cuda.synchronize()
    g.close()
    return w


@pytest.mark.parametrize("bc", FACES)
@pytest.mark.parametrize("order", [2, 4])
@pytest.mark.parametrize("n,nvec,spp", [((208, 160), 1, 25), ((209, 161), 1, 26), ((300, 250), 2, 41),
                                        ((517, 389), 4, 30), ((383, 319), 4, 34), ((700, 600), 1, 23),
                                        ((1000, 700), 1, 29), ((4000, 11), 1, 24), ((9, 5003), 1, 21),
                                        ((255, 257), 7, 33), ((1023, 641), 1, 22)])
def test_equals_blocked(ew, n, nvec, spp, order, bc):
    assert torch.equal(_apply(ew, n, order, bc, nvec, 0, spp), _apply(ew, n, order, bc, nvec, 2, spp))


def test_exchange_timeout_is_reported(ew, monkeypatch):
    n = (300, 250)
    g = ew.ew_grid_create(2, n, (1.0, 0.8), order=4, prec="fp32")
    p = ew.filter_params(40.0)
    v = torch.tensor(ew_inputs.uniform_pm1(14, g.size), dtype=torch.float32, device="cuda")
    w, ref = torch.empty_like(v), torch.empty_like(v)
    ew.ew_filter_apply(g, p, v, ref)
    monkeypatch.setenv("EW_TEST_RB2D_STALL", "1")
    ew.ew_filter_apply(g, p, v, w)
    monkeypatch.delenv("EW_TEST_RB2D_STALL")
    with pytest.raises(ew.EWError) as e:
        ew.ew_rayleigh(g, v)
    assert e.value.status == 6
    ew.ew_filter_apply(g, p, v, w)
    ew.ew_rayleigh(g, v)
    assert torch.equal(w, ref)
    g.close()
