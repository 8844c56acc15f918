"""Which kernels solve 2D shapes at the edges of the on-chip forms' ranges: the form that measured faster on each side,
and the bits of the blocked kernels either way."""
import pytest
import torch

import ew_inputs

pytestmark = pytest.mark.gpu


def _solve(n, order, prec, nvec, bc, spp):
    import __graft_entry__
    __graft_entry__.build()
    import paper_2507_18282_gb300 as ew
    rho = (4.0 if order == 2 else 16.0 / 3.0) * ((n[0] + 1) ** 2 + (n[1] + 1) ** 2)
    g = ew.ew_grid_create(2, n, (1.0, 1.0), order=order, prec=prec, bc=list(bc))
    v = torch.tensor(ew_inputs.uniform_pm1(29, g.size * nvec), dtype=g.dtype, device="cuda")
    outs = []
    for tb in (0, 2):
        p = ew.filter_params(3.14159 * rho**0.5 / (0.8 * spp), steps_per_period=spp, temporal_block=tb)
        outs.append(torch.full_like(v, float("nan")))
        ew.ew_filter_apply(g, p, v, outs[-1], nvec=nvec)
        if tb == 0:
            kernel = ew.tb2d_choice(g, nvec)["kernel"]
    torch.cuda.synchronize()
    g.close()
    assert torch.equal(outs[0], outs[1])
    return kernel


@pytest.mark.parametrize("n,order,prec,nvec,kernel", [
    ((240, 250), 4, "fp64", 1, "k_resident2d_cluster"), ((241, 249), 4, "fp64", 1, "k_step_tb2d"),
    ((255, 255), 2, "fp64", 1, "k_resident2d_cluster"), ((444, 91), 4, "fp32x2", 14, "k_resident2d_cluster"),
    ((444, 91), 4, "fp32x2", 15, "k_step_tb2d"), ((59, 593), 4, "fp32x2", 16, "k_resident2d_cluster")])
def test_cluster_or_blocked(n, order, prec, nvec, kernel):
    assert _solve(n, order, prec, nvec, "DDDD", 20).startswith(kernel)


@pytest.mark.parametrize("n,nvec,bc,spp,kernel", [
    ((446, 754), 4, "DDDD", 40, "k_step_"), ((446, 754), 4, "DDDD", 200, "k_persist2d"),
    ((446, 752), 4, "NDDD", 40, "k_persist2d"), ((268, 425), 6, "DDDD", 40, "k_persist2d")])
def test_cooperative_or_blocked(n, nvec, bc, spp, kernel):
    assert _solve(n, 4, "fp32", nvec, bc, spp).startswith(kernel)
