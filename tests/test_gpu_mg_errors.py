"""A launch that fails on a 3D FP32 multigrid level ends the call with its error: the residual, the damped-Jacobi
sweep and the colour sweep, in a single solve, a wave-solve and the smoother's training (a hook stands for the failed
launch, on the host).  The next call works again."""
import pytest
import torch

import ew_inputs

pytestmark = pytest.mark.gpu
EW_ECUDA = 3


@pytest.fixture(scope="module")
def ew():
    import __graft_entry__
    __graft_entry__.build()
    import paper_2507_18282_gb300 as ew
    return ew


@pytest.mark.parametrize("mode,red_black,learned", [(0, 0, 0), (1, 0, 0), (2, 1, 0), (0, 0, 1)])
def test_failed_launch_is_reported(ew, monkeypatch, mode, red_black, learned):
    n = (47, 31, 63)
    g = ew.ew_grid_create(3, n, (1.0, 1.0, 1.0), order=4, prec="fp32")
    b = torch.tensor(ew_inputs.uniform_pm1(31, g.size), dtype=torch.float32, device="cuda")
    w = torch.tensor(0.05 * ew_inputs.uniform_pm1(32, 432), dtype=torch.float32, device="cuda")
    mg = ew.mg_params(max_cycles=2, red_black=red_black, learned_levels=learned, weights=w if learned else None)
    p = ew.filter_params(12.0, steps_per_period=10, scheme="implicit", mg=mg)
    for call in (lambda: ew.ew_implicit_step_mg(g, 1e-3, b, torch.zeros_like(b), mg),
                 lambda: ew.ew_filter_apply(g, p, b, torch.empty_like(b))):
        monkeypatch.setenv("EW_TEST_MG_PLANE_FAIL", str(mode))
        with pytest.raises(ew.EWError) as e:
            call()
        assert e.value.status == EW_ECUDA
        monkeypatch.delenv("EW_TEST_MG_PLANE_FAIL")
        call()
    if mode == 0:
        monkeypatch.setenv("EW_TEST_MG_PLANE_FAIL", "0")
        with pytest.raises(ew.EWError) as e:
            ew.ew_smoother_train(g, 1e-3, w, steps=2, samples=2)
        assert e.value.status == EW_ECUDA
    torch.cuda.synchronize()
    g.close()
