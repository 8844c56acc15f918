"""Power iteration on a grid handle whose page-locked staging buffer has to grow for the filter weights (N_t of several
10,000) during the first application: the same numbers, bit for bit, as on a handle whose buffer is large already."""
import numpy as np
import pytest
import torch

import ew_inputs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec", ["fp32", "fp64"])
def test_fresh_handle(prec):
    import __graft_entry__
    __graft_entry__.build()
    import paper_2507_18282_gb300 as ew
    runs = []
    for grow_first in (True, False):
        g = ew.ew_grid_create(2, (20, 17), (1.0, 1.0), order=2, prec=prec)
        p = ew.filter_params(9.0, num_periods=3, steps_per_period=12000)
        v = torch.tensor(ew_inputs.uniform_pm1(91, g.size), dtype=g.dtype, device="cuda")
        if grow_first:
            ew.ew_filter_apply(g, ew.filter_params(9.0, num_periods=6, steps_per_period=12000), v, torch.empty_like(v))
        betas, done, lam = ew.ew_power_iteration(g, p, v, 3)
        runs.append((betas, lam, v.cpu().numpy()))
        assert done == 3
        g.close()
    for a, b in zip(*runs):
        assert np.array_equal(a, b)
