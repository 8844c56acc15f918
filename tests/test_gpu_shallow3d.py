"""Fourth-order FP32 3D boxes of a few planes, where one vector takes the one-step kernel and several (or eight planes)
the blocked one: the same bits at every temporal depth, and the launches each is expected to make."""
import numpy as np
import pytest
import torch

import ew_inputs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,nvec", [((5, 5, 5), 1), ((40, 33, 6), 1), ((40, 33, 7), 1), ((40, 33, 8), 1), ((70, 9, 1), 1),
                                    ((40, 33, 6), 2)])
def test_route_and_bits(n, nvec):
    import __graft_entry__
    __graft_entry__.build()
    import paper_2507_18282_gb300 as ew
    L, spp = (1.0, 0.9, 0.8), 13
    g = ew.ew_grid_create(3, n, L, order=4, prec="fp32", bc=list("NDDDDN"))
    blocked = g.n[2] >= 8 or nvec > 1  # active planes: the Neumann face's wall is one of them
    omega = 2.0 * np.pi * 0.5 * np.sqrt(16.0 / 3.0 * sum(((m + 1) / l) ** 2 for m, l in zip(n, L))) / (0.8 * spp)
    v = torch.tensor(ew_inputs.uniform_pm1(81, g.size * nvec), dtype=torch.float32, device="cuda")
    outs = []
    for tb in (1, 0, 2):
        p = ew.filter_params(omega, steps_per_period=spp, temporal_block=tb)
        outs.append(torch.full_like(v, float("nan")))
        ew.ew_profile_enable(True)
        ew.ew_filter_apply(g, p, v, outs[-1], nvec=nvec)
        launches = ew.ew_profile_read()["fused_launches"]
        ew.ew_profile_enable(False)
        steps = spp - 1
        assert launches == (steps * nvec if tb == 1 or not blocked else (steps + 1) // 2), (tb, launches)
    assert torch.equal(outs[0], outs[1]) and torch.equal(outs[0], outs[2])
    g.close()
