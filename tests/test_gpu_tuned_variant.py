"""ew_tuned_variant answers for every 2D shape that the blocked kernels or their on-chip forms have solved, and only
then; grids that one CTA holds stay refused."""
import pytest
import torch

import ew_inputs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,order,prec,nvec,kernel", [
    ((519, 387), 4, "fp32", 4, "k_persist2d<2"), ((301, 253), 2, "fp32", 1, "k_persist2d<1"),
    ((149, 151), 2, "fp32", 1, "k_resident2d_cluster<float, 1"), ((103, 157), 4, "fp64", 1, "k_resident2d_cluster<double, 2"),
    ((131, 97), 2, "fp32x2", 2, "k_resident2d_cluster<dd, 1"), ((1501, 1203), 4, "fp32", 1, "k_step_"),
    ((401, 399), 2, "fp64", 1, "k_step_tb2d<double"), ((61, 59), 2, "fp32", 1, None)])
def test_variant_of_the_last_solve(n, order, prec, nvec, kernel):
    import __graft_entry__
    __graft_entry__.build()
    import paper_2507_18282_gb300 as ew
    g = ew.ew_grid_create(2, n, (1.0, 0.8), order=order, prec=prec)
    assert ew.tb2d_choice(g, nvec) is None
    v = torch.tensor(ew_inputs.uniform_pm1(23, g.size * nvec), dtype=g.dtype, device="cuda")
    ew.ew_filter_apply(g, ew.filter_params(30.0), v, torch.empty_like(v), nvec=nvec)
    torch.cuda.synchronize()
    c = ew.tb2d_choice(g, nvec)
    if kernel is None:
        assert c is None
    else:
        assert c["kernel"].startswith(kernel) and c["depth"] >= 1
        assert 1 <= c["tile"][0] <= max(n) and 1 <= c["tile"][1] <= max(n)
    assert ew.tb2d_choice(g, nvec + 1) is None
    g.close()
