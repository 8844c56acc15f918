"""Second-order FP32 3D wave-solves blocked over time: the 32 x 32 and the 64 x 32 regions at each depth, chosen by hand
(the tuner's choice depends on timing), give the same bits, and stay within 4 N_t eps32 |v| of the FP64 oracle, the
bound of the other FP32 wave-solve tests.  Boxes narrower than, as wide as and wider than either region's owned tile,
few planes, N_t no multiple of the depth, each face kind."""
import numpy as np
import pytest
import torch

import ew_inputs
from oracle import oracle as O

pytestmark = pytest.mark.gpu
EPS32 = float(np.finfo(np.float32).eps)


@pytest.mark.parametrize("n,nvec,bc", [((27, 91, 33), 3, "DDDDDD"), ((26, 28, 70), 1, "NDDNDD"), ((33, 29, 130), 2, "DDNNDN"),
                                       ((3, 40, 20), 2, "DDDDDD"), ((122, 45, 9), 2, "DDDDNN"), ((24, 56, 41), 1, "NNNNNN")])
def test_regions_agree(monkeypatch, n, nvec, bc):
    import __graft_entry__
    __graft_entry__.build()
    import paper_2507_18282_gb300 as ew
    L, spp = (1.0, 1.2, 0.8), 15
    g = ew.ew_grid_create(3, n, L, order=2, prec="fp32", bc=list(bc))
    omega = 2.0 * np.pi * 0.5 * np.sqrt(4.0 * sum(((m + 1) / l) ** 2 for m, l in zip(n, L))) / (0.8 * spp)
    p = ew.filter_params(omega, steps_per_period=spp)
    v = torch.tensor(ew_inputs.uniform_pm1(71, g.size * nvec), dtype=torch.float32, device="cuda")
    outs = {}
    for region in ("wide", "narrow"):
        for depth in (2, 3, 4):
            monkeypatch.setenv("EW_TB3D_VARIANT", "%s:%d" % (region, depth))
            outs[region, depth] = torch.full_like(v, float("nan"))
            ew.ew_filter_apply(g, p, v, outs[region, depth], nvec=nvec)
    torch.cuda.synchronize()
    first = outs["wide", 2]
    for key, w in outs.items():
        assert torch.equal(first, w), key
    og, prm = O.Grid(n, L, 2, list(bc)), O.filter_params(omega, 1, spp)
    for q in {0, nvec - 1}:
        x = v[q * g.size:(q + 1) * g.size].double().cpu().numpy()
        y = first[q * g.size:(q + 1) * g.size].double().cpu().numpy()
        assert np.linalg.norm(y - O.filter_explicit(og, prm, x)) <= 4 * spp * EPS32 * np.linalg.norm(x)
    g.close()


@pytest.mark.parametrize("text", ["wide:5", "narrow:1", "narrow", "2", "wide:"])
def test_bad_override(monkeypatch, text):
    import __graft_entry__
    __graft_entry__.build()
    import paper_2507_18282_gb300 as ew
    g = ew.ew_grid_create(3, (27, 30, 31), (1.0, 1.0, 1.0), order=2, prec="fp32")
    v = torch.zeros(g.size, device="cuda")
    monkeypatch.setenv("EW_TB3D_VARIANT", text)
    with pytest.raises(ew.EWError) as e:
        ew.ew_filter_apply(g, ew.filter_params(10.0), v, torch.empty_like(v))
    assert e.value.status == 1
    g.close()
