"""Second-order FP32 3D wave-solves on narrow and shallow boxes (32 x 32 regions beside the 64 x 32 ones): every depth and
the tuned choice give the bits of the one-step kernels."""
import pytest
import torch

import ew_inputs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,nvec,bc", [((27, 91, 33), 3, "DDDDDD"), ((32, 65, 70), 1, "NDDNDD"), ((33, 29, 130), 2, "DDDDDD"),
                                       ((1, 40, 20), 2, "DDDDDD"), ((122, 45, 9), 2, "DDDDNN")])
def test_bits(n, nvec, bc):
    import __graft_entry__
    __graft_entry__.build()
    import paper_2507_18282_gb300 as ew
    g = ew.ew_grid_create(3, n, (1.0, 1.2, 0.8), order=2, prec="fp32", bc=list(bc))
    v = torch.tensor(ew_inputs.uniform_pm1(71, g.size * nvec), dtype=torch.float32, device="cuda")
    outs = []
    for tb in (1, 0, 2, 3, 4):
        p = ew.filter_params(14.0, temporal_block=tb)
        w = torch.full_like(v, float("nan"))
        ew.ew_filter_apply(g, p, v, w, nvec=nvec)
        outs.append(w)
    torch.cuda.synchronize()
    scale = float(outs[0].abs().max())
    for w in outs[2:]:  # the blocked forms agree with one another, whatever the depth and the region
        assert torch.equal(outs[1], w)
    # the one-step kernel sums a point's neighbours in another order: rounding, 64 operations a step at most
    assert float((outs[0] - outs[1]).abs().max()) <= 64 * 2.0**-24 * 200 * scale
    g.close()
