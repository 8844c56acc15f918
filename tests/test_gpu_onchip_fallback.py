"""On-chip wave-solves where the device cannot hold their CTAs together (hooks stand for a partitioned GPU): clusters
of at most 8, 4, 2 or 1 CTAs, or none, and a cooperative launch that is refused.  The call takes the next form and
gives the same bits."""
import pytest
import torch

import ew_inputs

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ew():
    import __graft_entry__
    __graft_entry__.build()
    import paper_2507_18282_gb300 as ew
    return ew


def _solve(ew, n, order, prec, nvec, bc):
    g = ew.ew_grid_create(2, n, (1.0, 0.8), order=order, prec=prec, bc=list(bc))
    p = ew.filter_params(12.0)
    v = torch.tensor(ew_inputs.uniform_pm1(17, g.size * nvec), dtype=g.dtype, device="cuda")
    w = torch.full_like(v, float("nan"))
    ew.ew_filter_apply(g, p, v, w, nvec=nvec)
    torch.cuda.synchronize()
    g.close()
    return w


@pytest.mark.parametrize("largest", [8, 4, 2, 1, 0])
@pytest.mark.parametrize("n,order,prec,nvec", [((63, 63), 2, "fp64", 1), ((63, 64), 4, "fp32", 3), ((50, 61), 4, "fp32x2", 1),
                                               ((129, 130), 4, "fp32", 1), ((97, 120), 2, "fp64", 2),
                                               ((90, 140), 2, "fp32x2", 1)])
def test_smaller_clusters(ew, monkeypatch, n, order, prec, nvec, largest):
    ref = _solve(ew, n, order, prec, nvec, "NDDD")
    monkeypatch.setenv("EW_TEST_MAX_CLUSTER", str(largest))
    assert torch.equal(_solve(ew, n, order, prec, nvec, "NDDD"), ref)


@pytest.mark.parametrize("n,order,nvec", [((300, 250), 4, 1), ((517, 389), 2, 3)])
def test_refused_cooperative_launch(ew, monkeypatch, n, order, nvec):
    ref = _solve(ew, n, order, "fp32", nvec, "DDND")
    monkeypatch.setenv("EW_TEST_COOP_TOO_LARGE", "1")
    assert torch.equal(_solve(ew, n, order, "fp32", nvec, "DDND"), ref)
