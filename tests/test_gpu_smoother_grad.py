"""Weight gradient of the learned smoother at the edges of its kernel's tiles (32 x 8 x 4 points with a halo of one,
three columns a step): one point, exact tiles, one point more or less on each axis, several tiles a CTA.

Bounds, per component, against the FP64 oracle (weights and residual BF16 values on both sides): dW2 inherits the
hidden activations' one BF16 rounding, u sum |gy| |h| with u = 2^-8; both layers' sums keep about 48 bits, so what is
left is the rounding of dh (27 terms, 27 2^-24 sum |W2| |gy| |r|) and of the stored result."""
import numpy as np
import pytest
import torch

import ew_inputs
from oracle import oracle as O

pytestmark = pytest.mark.gpu
U_BF16, EPS = 2.0 ** -8, 2.0 ** -24


def _bf16(x):
    return torch.tensor(np.asarray(x), dtype=torch.float32).to(torch.bfloat16).double().numpy()


def _taps_sum(a, b):
    """sum_x a(x) b(x + o) for the 27 offsets, b zero outside the box."""
    bp = np.pad(b, 1)
    nz, ny, nx = a.shape
    return np.array([np.sum(a * bp[dz:dz + nz, dy:dy + ny, dx:dx + nx])
                     for dz in range(3) for dy in range(3) for dx in range(3)])


@pytest.mark.parametrize("prec", ["fp32", "fp64"])
@pytest.mark.parametrize("n", [(1, 1, 1), (2, 3, 1), (32, 8, 4), (33, 9, 5), (31, 7, 3), (35, 17, 1), (64, 40, 26),
                               (97, 66, 60)])
def test_gradient_tile_edges(n, prec):
    import __graft_entry__
    __graft_entry__.build()
    import paper_2507_18282_gb300 as ew
    g = ew.ew_grid_create(3, n, (1.0, 1.0, 1.0), order=4, prec=prec)
    N = g.size
    w = _bf16(ew_inputs.learned_init(71, 0.3))
    r = _bf16(ew_inputs.uniform_pm1(72, N))
    gy = ew_inputs.uniform_pm1(73, N).astype(np.float32).astype(np.float64)
    dt = torch.float32 if prec == "fp32" else torch.float64
    grad = torch.empty(432, dtype=torch.float32, device="cuda")
    ew.ew_smoother_backward(g, torch.tensor(w, dtype=torch.float32, device="cuda"),
                            torch.tensor(r, dtype=dt, device="cuda"), torch.tensor(gy, dtype=dt, device="cuda"), grad)
    torch.cuda.synchronize()
    hid, _ = O.conv_net_forward(n, w, r)
    ref, _ = O.conv_net_backward(n, w, r, hid, gy)
    shape = (n[2], n[1], n[0])
    ar, ag = np.abs(r).reshape(shape), np.abs(gy).reshape(shape)
    bound = np.zeros(432)
    for c in range(8):
        bound[216 + c * 27:216 + (c + 1) * 27] = U_BF16 * _taps_sum(ag, np.abs(hid[c * N:(c + 1) * N]).reshape(shape))
        adh = np.zeros(shape)  # sum_o |W2[c][o]| |gy(y - o)|
        gp = np.pad(ag, 1)
        for t in range(27):
            dz, dy, dx = 2 - t // 9, 2 - (t // 3) % 3, 2 - t % 3
            adh += abs(w[216 + c * 27 + t]) * gp[dz:dz + n[2], dy:dy + n[1], dx:dx + n[0]]
        bound[c * 27:(c + 1) * 27] = 28 * EPS * _taps_sum(adh, ar)
    bound += 2 * EPS * np.abs(ref) + 1e-30
    diff = np.abs(grad.cpu().double().numpy() - ref)
    assert np.all(diff <= bound), float(np.max(diff / bound))
    g.close()
