"""The work whose time is tracked: applications of the filter operator S and the calls around it.

A user of this library applies S (one wave-solve) to start vectors and Krylov blocks on boxes and curvilinear
grids, in FP32, FP64 and double-FP32 pairs, explicitly and implicitly, one problem at a time or many at once, trains
the learned smoother, and runs the eigen-solver.  Every case goes through the public entry points with buffers and
handles such a program keeps; inputs are uniform [-1, 1) on the active points, the start vectors of the method.

`exact` restates each case in 64-bit torch (dense stencils by index, sine transforms, dense coarse solves) without
the library's code.
"""
from __future__ import annotations

import math
import random

import numpy as np
import torch

import paper_2507_18282_gb300 as ew

CFL = 0.8


# ---------------------------------------------------------------------------------------------------------------
# the cases
# ---------------------------------------------------------------------------------------------------------------
def listed():
    return [
        # the smallest problem in use: one vector on the 63^2 unit square in FP64; launches and latency
        dict(name="square63_fp64", kind="box", n="63x63", length="1.0x1.0", order=2, prec="fp64", omega=20.0,
             periods=1, nvec=1, bc="DDDD"),
        # an ordinary Krylov block on a ragged mid-size box with a symmetry plane
        dict(name="box2d_517x389_sym_block4", kind="box", n="517x389", length="1.0x0.75", order=4, prec="fp32",
             omega=40.0, periods=1, nvec=4, bc="NDDD"),
        # the headline wave-solve of the benchmark: a block of 16 vectors on 2047 x 3071
        dict(name="rect2d_2047x3071_block16", kind="box", n="2047x3071", length="1.0x1.5", order=4, prec="fp32",
             omega=150.0, periods=1, nvec=16, bc="DDDD"),
        # the refinement's images: a block of 8 vectors in double-FP32 pairs at half that resolution
        dict(name="rect2d_1023x1535_pairs_block8", kind="box", n="1023x1535", length="1.0x1.5", order=4,
             prec="fp32x2", omega=75.0, periods=1, nvec=8, bc="DDDD"),
        # the large 3D cube of the benchmark, one vector, second order
        dict(name="cube511_order2", kind="box", n="511x511x511", length="1.0x1.0x1.0", order=2, prec="fp32",
             omega=60.0, periods=1, nvec=1, bc="DDDDDD"),
        # fourth-order 3D on a ragged box, a block of two vectors, explicit
        dict(name="box3d_191x161x143_order4", kind="box", n="191x161x143", length="1.0x0.85x0.75", order=4,
             prec="fp32", omega=20.0, periods=1, nvec=2, bc="DDDDDD"),
        # many uneven boxes in one call, as a batched eigen-solve asks for
        dict(name="batched_64_boxes", kind="batched", count=64, n_min=255, n_max=2047, order=2, w_min=10.0,
             w_max=200.0, boxes=2507),
        # a curvilinear grid (warped unit square) at the benchmark's size
        dict(name="mapped2d_2047", kind="mapped", n="2047x2047", prec="fp32", eps=0.1, omega=80.0, periods=1, nvec=1),
        # the implicit scheme on a square in FP64, every system solved to 1e-10 with red-black smoothing
        dict(name="square1023_implicit_fp64", kind="implicit", n="1023x1023", length="1.0x1.0", order=2, prec="fp64",
             omega=12.0, periods=1, spp=10, cycles=30, rtol=1e-10, learned=0, red_black=1, guess="previous"),
        # the implicit order-4 cube with the learned smoother on the finest level, two V(2,2) cycles per system
        dict(name="cube255_implicit_learned", kind="implicit", n="255x255x255", length="1.0x1.0x1.0", order=4,
             prec="fp32", omega=80.0, periods=1, spp=10, cycles=2, rtol=0.0, learned=1, red_black=0, guess="rhs"),
        # one training evaluation of the learned smoother: the network's output and its weights' gradient
        dict(name="smoother_train_127", kind="smoother", n="127x127x127", order=4, omega=40.0),
        # a whole eigen-solve: FP32 Krylov-Schur stage, refinement with double-FP32 images
        dict(name="eigs2d_383x319_refined", kind="eigs", n="383x319", length="1.0x0.83", order=4, omega=30.0,
             wanted=8, krylov=32, block=4),
    ]


def _logint(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _text(values):
    return "x".join(str(v) for v in values)


def _open(case):
    """The case with its sizes (texts such as "517x389") as lists of numbers."""
    out = dict(case)
    if "n" in out:
        out["n"] = [int(m) for m in out["n"].split("x")]
    if "length" in out:
        out["length"] = [float(l) for l in out["length"].split("x")]
    return out


def _rho(length, n, order):
    return (4.0 if order == 2 else 16.0 / 3.0) * sum(((m + 1) / l) ** 2 for m, l in zip(n, length))


def _omega_for(length, n, order, spp):
    return round(2.0 * math.pi * 0.5 * math.sqrt(_rho(length, n, order)) / (CFL * spp), 4)


def _draw_box2d(rng):
    prec = rng.choice(["fp32", "fp32", "fp32", "fp64", "fp32x2"])
    cap = 8e9 if prec == "fp32" else 6e8
    while True:
        n = [_logint(rng, 31, 3071), _logint(rng, 31, 3071)]
        spp, nvec = _logint(rng, 12, 240), rng.choice([1, 1, 2, 3, 4, 6, 8, 16])
        if n[0] * n[1] * spp * nvec <= cap:
            break
    length = [1.0, round(rng.uniform(0.5, 2.0), 3)]
    order = rng.choice([2, 4])
    bc = rng.choice(["DDDD", "DDDD", "NDDD", "DDDN", "NDNN"])
    return dict(kind="box", n=n, length=length, order=order, prec=prec, omega=_omega_for(length, n, order, spp),
                periods=1, nvec=nvec, bc=bc)


def _draw_box3d(rng):
    while True:
        n = [_logint(rng, 24, 511) for _ in range(3)]
        spp, nvec = _logint(rng, 12, 120), rng.choice([1, 1, 2, 4, 6])
        if n[0] * n[1] * n[2] * spp * nvec <= 3e9:
            break
    length = [1.0, round(rng.uniform(0.6, 1.5), 3), round(rng.uniform(0.6, 1.5), 3)]
    order = rng.choice([2, 4])
    bc = rng.choice(["DDDDDD", "DDDDDD", "NDDDDD", "DDDDNN"])
    return dict(kind="box", n=n, length=length, order=order, prec="fp32", omega=_omega_for(length, n, order, spp),
                periods=1, nvec=nvec, bc=bc)


def _draw_batched(rng):
    return dict(kind="batched", count=_logint(rng, 4, 64), n_min=127, n_max=_logint(rng, 255, 1535),
                order=rng.choice([2, 2, 4]), w_min=20.0, w_max=200.0, boxes=rng.randrange(1 << 20))


def _draw_mapped(rng):
    n = [_logint(rng, 63, 2047), _logint(rng, 63, 2047)]
    nvec = rng.choice([1, 2, 4])
    if n[0] * n[1] > 1 << 20:
        nvec = 1
    return dict(kind="mapped", n=n, prec=rng.choice(["fp32", "fp32", "fp32", "fp64"]),
                eps=round(rng.uniform(0.0, 0.12), 3), omega=round(max(n) * rng.uniform(0.03, 0.08), 3), periods=1,
                nvec=nvec)


def _draw_implicit(rng):
    order = rng.choice([2, 4])
    if rng.random() < 0.5:  # 2D, systems to a tolerance
        k = rng.randrange(4, 8)
        n = [rng.choice([4, 5, 6, 7, 8]) * 2 ** k - 1, rng.choice([4, 5, 6, 7, 8]) * 2 ** k - 1]
        return dict(kind="implicit", n=n, length=[1.0, round((n[1] + 1) / (n[0] + 1), 6)], order=order,
                    prec=rng.choice(["fp64", "fp64", "fp32"]), omega=round(rng.uniform(8.0, 24.0), 3), periods=1,
                    spp=10, cycles=30, rtol=1e-5, learned=0, red_black=rng.choice([0, 1]),
                    guess=rng.choice(["rhs", "previous"]))
    k = rng.randrange(3, 6)  # 3D, a fixed number of cycles
    n = [rng.choice([4, 5, 6, 7]) * 2 ** k - 1 for _ in range(3)]
    return dict(kind="implicit", n=n, length=[1.0] + [round((m + 1) / (n[0] + 1), 6) for m in n[1:]], order=order,
                prec="fp32", omega=round(n[0] * 0.31, 3), periods=1, spp=10, cycles=rng.choice([2, 3]), rtol=0.0,
                learned=rng.choice([0, 1]), red_black=0, guess="rhs")


def _draw_smoother(rng):
    n = [_logint(rng, 31, 191) for _ in range(3)]
    return dict(kind="smoother", n=n, order=rng.choice([2, 4]), omega=round(n[0] * 0.31, 3))


def _draw_eigs(rng):
    n = [_logint(rng, 160, 420), _logint(rng, 160, 420)]
    return dict(kind="eigs", n=n, length=[1.0, round(rng.uniform(0.61, 1.37), 3)], order=rng.choice([2, 4]),
                omega=round(rng.uniform(22.0, 36.0), 2), wanted=rng.choice([4, 6, 8]), krylov=32, block=4)


def draw(rng: random.Random):
    """One more case of the ranges above: log-uniform sizes, ragged ones among them."""
    case = rng.choice([_draw_box2d, _draw_box2d, _draw_box2d, _draw_box3d, _draw_box3d, _draw_batched, _draw_mapped,
                       _draw_implicit, _draw_implicit, _draw_smoother, _draw_eigs])(rng)
    return {k: _text(v) if isinstance(v, list) else v for k, v in case.items()}


# ---------------------------------------------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------------------------------------------
def _uniform(count, seed, dtype, scale=1.0):
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed)
    return torch.empty(count, dtype=dtype, device="cuda").uniform_(-scale, scale, generator=gen)


def _dtype(prec):
    return torch.float32 if prec == "fp32" else torch.float64


def _boxes(case):
    """Side lengths, sizes and frequencies of the uneven boxes: the case fixes them."""
    rng = random.Random(case["boxes"])
    out = []
    for _ in range(case["count"]):
        lx, ly = rng.uniform(0.5, 2.0), rng.uniform(0.5, 2.0)
        n = min(max(_logint(rng, case["n_min"], case["n_max"]), case["n_min"]), case["n_max"])
        out.append(dict(n=[n, n], length=[lx, ly], order=case["order"], prec="fp32",
                        omega=rng.uniform(case["w_min"], case["w_max"]), periods=1, nvec=1, bc="DDDD"))
    return out


def _warped_vertices(n, eps):
    r, s = np.linspace(0.0, 1.0, n[0] + 2), np.linspace(0.0, 1.0, n[1] + 2)
    R, S = np.meshgrid(r, s)
    x = R + eps * np.sin(np.pi * R) * np.cos(np.pi * S)
    y = S + eps * np.sin(np.pi * S) * np.cos(np.pi * R)
    return np.ascontiguousarray(np.stack([x, y], axis=-1))


def _half_dt2(omega, spp):
    """dt^2 / 2 of the implicit scheme at the adjusted frequency."""
    s = math.sin(math.pi / spp)
    w = omega * math.pi / spp * math.sqrt((1.0 - 2.0 * s * s) / (s * s))
    return 0.5 * (2.0 * math.pi / w / spp) ** 2, w


def _smoother_weights(case, seed, length):
    """A convergent smoother that uses every tap: near the damped-Jacobi correction, each weight perturbed."""
    a, _ = _half_dt2(case["omega"], 10)
    d0 = 2.0 if case["order"] == 2 else 2.5
    centre = 0.8 / (1.0 + a * sum(d0 * ((m + 1) / l) ** 2 for m, l in zip(case["n"], length)))
    w = _uniform(432, seed, torch.float32, 0.02)
    w[216:] *= centre
    w[13] += 1.0
    w[216 + 13] += centre
    return w


def prepare(case, seed):
    case = _open(case)
    kind = case["kind"]
    if kind == "box":
        g = ew.ew_grid_create(len(case["n"]), case["n"], case["length"], order=case["order"], prec=case["prec"],
                              bc=list(case["bc"]))
        p = ew.filter_params(case["omega"], num_periods=case["periods"], cfl=CFL)
        v = _uniform(g.size * case["nvec"], seed, g.dtype)
        return dict(kind=kind, g=g, p=p, v=v, w=torch.empty_like(v), nvec=case["nvec"])
    if kind == "batched":
        boxes = _boxes(case)
        gs = [ew.ew_grid_create(2, b["n"], b["length"], order=b["order"], prec="fp32") for b in boxes]
        ps = [ew.filter_params(b["omega"], num_periods=1, cfl=CFL) for b in boxes]
        vs = [_uniform(g.size, seed + 1000 * q, torch.float32) for q, g in enumerate(gs)]
        return dict(kind=kind, g=gs, p=ps, v=vs, w=[torch.empty_like(v) for v in vs])
    if kind == "mapped":
        g = ew.ew_grid_create_mapped(case["n"], _warped_vertices(case["n"], case["eps"]), prec=case["prec"])
        p = ew.filter_params(case["omega"], num_periods=case["periods"], cfl=CFL)
        v = _uniform(g.size * case["nvec"], seed, g.dtype)
        return dict(kind="box", g=g, p=p, v=v, w=torch.empty_like(v), nvec=case["nvec"])
    if kind == "implicit":
        g = ew.ew_grid_create(len(case["n"]), case["n"], case["length"], order=case["order"], prec=case["prec"])
        wts = _smoother_weights(case, 432, case["length"]) if case["learned"] else None
        mg = ew.mg_params(pre=2, post=2, max_cycles=case["cycles"], rtol=case["rtol"], learned_levels=case["learned"],
                          weights=wts, red_black=bool(case["red_black"]), guess=case["guess"])
        p = ew.filter_params(case["omega"], num_periods=case["periods"], steps_per_period=case["spp"],
                             scheme="implicit", adjust_omega=True, mg=mg)
        v = _uniform(g.size, seed, g.dtype)
        return dict(kind="box", g=g, p=p, v=v, w=torch.empty_like(v), nvec=1)
    if kind == "smoother":
        g = ew.ew_grid_create(3, case["n"], [1.0, 1.0, 1.0], order=case["order"], prec="fp32")
        return dict(kind=kind, g=g, wts=_smoother_weights(case, seed + 1, [1.0, 1.0, 1.0]),
                    r=_uniform(g.size, seed, torch.float32), gy=_uniform(g.size, seed + 2, torch.float32),
                    y=torch.empty(g.size, dtype=torch.float32, device="cuda"),
                    grad=torch.empty(432, dtype=torch.float32, device="cuda"))
    if kind == "eigs":
        g = ew.ew_grid_create(2, case["n"], case["length"], order=case["order"], prec="fp32")
        p = ew.filter_params(case["omega"], num_periods=_eigs_periods(case), cfl=CFL)
        e = ew.eigs_params(case["wanted"], krylov_dim=case["krylov"], block=case["block"], refine_fp64=3)
        return dict(kind=kind, g=g, p=p, e=e, start=_uniform(g.size * case["block"], seed, torch.float64),
                    vecs=torch.empty(case["wanted"] * g.size, dtype=torch.float64, device="cuda"))
    raise ValueError(kind)


def _eigs_periods(case):
    """N_p by the library's own estimate, the choice a user takes."""
    g = ew.ew_grid_create(2, case["n"], case["length"], order=case["order"], prec="fp32")
    n_p, _ = ew.ew_choose_num_periods(g, ew.filter_params(case["omega"], cfl=CFL), case["wanted"], case["krylov"],
                                      max_periods=64)
    g.close()
    return n_p


# ---------------------------------------------------------------------------------------------------------------
# one pass
# ---------------------------------------------------------------------------------------------------------------
def run(state):
    kind = state["kind"]
    if kind == "box":
        ew.ew_filter_apply(state["g"], state["p"], state["v"], state["w"], nvec=state["nvec"])
        return state["w"]
    if kind == "batched":
        ew.ew_filter_apply_batched(state["g"], state["p"], state["v"], state["w"])
        return state["w"]
    if kind == "smoother":
        ew.ew_smoother_forward(state["g"], state["wts"], state["r"], state["y"])
        ew.ew_smoother_backward(state["g"], state["wts"], state["r"], state["gy"], state["grad"])
        return {"y": state["y"], "grad": state["grad"]}
    lam, _, _ = ew.ew_arnoldi_eigs(state["g"], state["p"], state["e"], start=state["start"], vecs=state["vecs"])
    # eigenvectors are defined up to sign: oriented along the first start vector
    n = state["g"].size
    vecs = state["vecs"].view(-1, n)
    sign = torch.where(vecs @ state["start"][:n] < 0, -1.0, 1.0).to(torch.float64)
    return {"lam": lam, "vecs": vecs * sign[:, None]}


# ---------------------------------------------------------------------------------------------------------------
# what a pass cannot do without
# ---------------------------------------------------------------------------------------------------------------
def _active(case):
    bc = case.get("bc", "DDDDDD")
    return [m + (bc[2 * a] == "N") + (bc[2 * a + 1] == "N") for a, m in enumerate(case["n"])]


def _spp(case):
    if "spp" in case:
        return case["spp"]
    dtmax = 2.0 / math.sqrt(_rho(case["length"], case["n"], case["order"]))
    return max(1, math.ceil(2.0 * math.pi / case["omega"] / (CFL * dtmax) - 1e-12))


def _box_work(case):
    N = math.prod(_active(case))
    es = 4 if case["prec"] == "fp32" else 8
    # per point and step: the Laplacian, D += lap, W += D, acc += c W
    flops = 5 + 3 * len(case["n"]) * (1 if case["order"] == 2 else 2)
    return dict(bytes=2 * N * case["nvec"] * es, flops=flops * N * case["nvec"] * _spp(case) * case["periods"])


def work(case):
    case = _open(case)
    kind = case["kind"]
    if kind == "box":
        return _box_work(case)
    if kind == "batched":
        each = [_box_work(b) for b in _boxes(case)]
        return dict(bytes=sum(e["bytes"] for e in each), flops=sum(e["flops"] for e in each))
    N = math.prod(case["n"])
    if kind == "mapped":
        es = 4 if case["prec"] == "fp32" else 8
        steps = math.ceil(2.0 * math.pi / case["omega"] / (CFL * 2.0 / math.sqrt(_mapped_rho_estimate(case))))
        # vectors in and out, six couplings a point; 9-point stencil, 1/J, D, W, acc
        return dict(bytes=es * N * (2 * case["nvec"] + 6), flops=24 * N * case["nvec"] * steps * case["periods"])
    if kind == "implicit":
        d = len(case["n"])
        es = 4 if case["prec"] == "fp32" else 8
        point = 5 + 3 * d * (1 if case["order"] == 2 else 2)  # one smoothing step or residual
        cycles = case["cycles"] if case["rtol"] == 0.0 else max(2, round(-math.log10(case["rtol"]) * 0.8))
        geom = 1.0 / (1.0 - 0.5 ** d)
        per_cycle = 5 * point * geom + (4 * 250 if case["learned"] else 0)
        return dict(bytes=2 * N * es, flops=int(N * (per_cycle * cycles + 3) * case["spp"] * case["periods"]))
    if kind == "smoother":
        # two 27-tap layers of 8 channels forward, the same again for the hidden layer, twice that for the gradient
        return dict(bytes=4 * (3 * N + 3 * 432), flops=N * (864 + 3 * 864))
    # eigs: at least a Krylov basis of wave-solves and its orthogonalisation
    N, m = math.prod(case["n"]), case["krylov"]
    flops = (5 + 6 * (1 if case["order"] == 2 else 2)) * N * _spp(case) * _eigs_periods(case) * m + 4 * N * m * m
    return dict(bytes=8 * N * (case["block"] + case["wanted"]), flops=flops)


def _mapped_rho_estimate(case):
    """The step limit's spectral bound of the warped square: twice the Cartesian one at most, for a small warp."""
    return 4.0 * sum((m + 1) ** 2 for m in case["n"]) * (1.0 + 3.0 * case["eps"])


# ---------------------------------------------------------------------------------------------------------------
# the same results in 64 bits, from plain torch
# ---------------------------------------------------------------------------------------------------------------
def _plan(omega, periods, spp):
    Nt = periods * spp
    Tf = periods * 2.0 * math.pi / omega
    dt = Tf / Nt
    alpha = math.tan(0.5 * omega * dt) / math.tan(omega * dt)
    sig = [0.5 * dt if n in (0, Nt) else dt for n in range(Nt + 1)]
    return Nt, dt, [2.0 / Tf * sig[n] * (math.cos(omega * n * dt) - 0.5 * alpha) for n in range(Nt + 1)]


def _reflect(n, lo, hi, off, dev):
    """Index and sign of the point `off` beyond each of n active points, by reflection about the walls."""
    wl, wu = (0 if lo == "N" else -1), (n - 1 if hi == "N" else n)
    idx, sgn = [], []
    for i in range(n):
        p, s = i + off, 1.0
        while p < wl or p > wu:
            if p < wl:
                p, s = 2 * wl - p, s * (1.0 if lo == "N" else -1.0)
            else:
                p, s = 2 * wu - p, s * (1.0 if hi == "N" else -1.0)
        if p < 0 or p >= n:
            p, s = i, 0.0
        idx.append(p)
        sgn.append(s)
    return torch.tensor(idx, device=dev), torch.tensor(sgn, dtype=torch.float64, device=dev)


class _Lap:
    """L_h on tensors (..., [nz,] ny, nx) with reflected walls."""

    def __init__(self, n, h, order, bc, dev):
        self.terms, self.c0 = [], 0.0
        for a, m in enumerate(n):
            i2 = 1.0 / h[a] ** 2
            w = {1: i2} if order == 2 else {1: 16.0 / 12.0 * i2, 2: -i2 / 12.0}
            for off, c in w.items():
                self.c0 -= 2.0 * c
                for s in (-off, off):
                    idx, sg = _reflect(m, bc[2 * a], bc[2 * a + 1], s, dev)
                    self.terms.append((-1 - a, idx, sg.view([-1] + [1] * a), c))

    def __call__(self, u):
        r = self.c0 * u
        for ax, idx, sg, c in self.terms:
            t = u.index_select(u.dim() + ax, idx)
            t *= sg
            r.add_(t, alpha=c)
        return r


def _leapfrog(lap, v, plan):
    Nt, dt, c = plan
    d = lap(v) * (0.5 * dt * dt)
    w = v + d
    acc = c[0] * v + c[1] * w
    for n in range(1, Nt):
        d.add_(lap(w), alpha=dt * dt)
        w += d
        acc.add_(w, alpha=c[n + 1])
    return acc


def _exact_box(case, v):
    n = _active(case)
    h = [l / (m + 1) for l, m in zip(case["length"], case["n"])]
    lap = _Lap(n, h, case["order"], case["bc"], v.device)
    u = v.double().view([case["nvec"]] + n[::-1])
    return _leapfrog(lap, u, _plan(case["omega"], case["periods"], _spp(case))).reshape(-1)


class _MappedLap:
    """The conservative 9-point operator of a vertex map, u = 0 on the boundary vertices."""

    def __init__(self, n, xy, dev):
        p1, p2 = n[0] + 2, n[1] + 2
        dr, ds = 1.0 / (n[0] + 1), 1.0 / (n[1] + 1)
        X = torch.tensor(xy, dtype=torch.float64, device=dev)

        def diff(a, axis, h):
            a = a.transpose(0, axis)
            out = torch.empty_like(a)
            out[1:-1] = (a[2:] - a[:-2]) / (2.0 * h)
            out[0] = (-3.0 * a[0] + 4.0 * a[1] - a[2]) / (2.0 * h)
            out[-1] = (3.0 * a[-1] - 4.0 * a[-2] + a[-3]) / (2.0 * h)
            return out.transpose(0, axis)

        xr, yr = diff(X[..., 0], 1, dr), diff(X[..., 1], 1, dr)
        xs, ys = diff(X[..., 0], 0, ds), diff(X[..., 1], 0, ds)
        J = xr * ys - xs * yr
        A11, A22, A12 = (xs ** 2 + ys ** 2) / J, (xr ** 2 + yr ** 2) / J, -(xr * xs + yr * ys) / J
        cx, cy, cxy = 1.0 / dr ** 2, 1.0 / ds ** 2, 1.0 / (4.0 * dr * ds)
        E, N, NE, SE = (torch.zeros(p2, p1, dtype=torch.float64, device=dev) for _ in range(4))
        E[:, :-1] = 0.5 * (A11[:, :-1] + A11[:, 1:]) * cx
        N[:-1] = 0.5 * (A22[:-1] + A22[1:]) * cy
        NE[:-1, :-1] = (A12[:-1, 1:] + A12[1:, :-1]) * cxy
        SE[1:, :-1] = -(A12[1:, 1:] + A12[:-1, :-1]) * cxy
        i = (slice(1, -1), slice(1, -1))
        w, s = (slice(1, -1), slice(0, -2)), (slice(0, -2), slice(1, -1))
        sw, nw = (slice(0, -2), slice(0, -2)), (slice(2, None), slice(0, -2))
        self.links = [(E[i], 0, 1), (E[w], 0, -1), (N[i], 1, 0), (N[s], -1, 0), (NE[i], 1, 1), (NE[sw], -1, -1),
                      (SE[i], -1, 1), (SE[nw], 1, -1)]
        self.rj = 1.0 / J[i]
        total = sum(c for c, _, _ in self.links)
        self.centre = -total
        self.rho = float(((total.abs() + sum(c.abs() for c, _, _ in self.links)) * self.rj).max())

    def __call__(self, u):
        up = torch.nn.functional.pad(u, (1, 1, 1, 1))
        ny, nx = u.shape[-2:]
        r = self.centre * u
        for c, dy, dx in self.links:
            r += c * up[..., 1 + dy:1 + dy + ny, 1 + dx:1 + dx + nx]
        return r * self.rj


def _exact_mapped(case, v):
    lap = _MappedLap(case["n"], _warped_vertices(case["n"], case["eps"]), v.device)
    spp = math.ceil(2.0 * math.pi / case["omega"] / (CFL * 2.0 / math.sqrt(lap.rho)) - 1e-12)
    u = v.double().view(case["nvec"], case["n"][1], case["n"][0])
    return _leapfrog(lap, u, _plan(case["omega"], case["periods"], spp)).reshape(-1)


def _sines(u, axis):
    """The orthonormal discrete sine transform (its own inverse) along an axis."""
    n = u.shape[axis]
    u = u.transpose(axis, -1)
    z = torch.zeros(u.shape[:-1] + (2 * (n + 1),), dtype=u.dtype, device=u.device)
    z[..., 1:n + 1] = u
    s = -torch.fft.fft(z).imag[..., 1:n + 1] * math.sqrt(2.0 / (n + 1))
    return s.transpose(axis, -1).contiguous()


def _symbol(n, h, order, dev):
    s = torch.sin(torch.arange(1, n + 1, dtype=torch.float64, device=dev) * (0.5 * math.pi / (n + 1))) ** 2
    return (4.0 * s + (4.0 / 3.0 * s * s if order == 4 else 0.0)) / h ** 2


def _implicit_solved(case, v, h, a, plan):
    """Every system solved exactly, mode by mode."""
    Nt, _, c = plan
    n = case["n"]
    u = v.double().view(n[::-1])
    for ax in range(len(n)):
        u = _sines(u, ax)
    lam2 = sum(_symbol(m, h[q], case["order"], v.device).view([-1] + [1] * q) for q, m in enumerate(n))
    m = 1.0 + a * lam2
    w0, w1 = torch.ones_like(m), 1.0 / m
    out = c[0] * w0 + c[1] * w1
    for k in range(1, Nt):
        w0, w1 = w1, 2.0 * w1 / m - w0
        out += c[k + 1] * w1
    u = u * out
    for ax in range(len(n)):
        u = _sines(u, ax)
    return u.reshape(-1)


class _Cycle:
    """The V(2,2) cycle: learned or damped-Jacobi smoothing, full weighting, linear interpolation, exact coarse solve."""

    def __init__(self, case, h, a, dev, wts):
        self.lv, n, h = [], list(case["n"]), list(h)
        d0 = 2.0 if case["order"] == 2 else 2.5
        while True:
            self.lv.append((n, _Lap(n, h, case["order"], "DD" * len(n), dev), 1.0 + a * sum(d0 / x ** 2 for x in h)))
            if any(m < 5 or m % 2 == 0 for m in n):
                break
            n, h = [(m - 1) // 2 for m in n], [2.0 * x for x in h]
        self.a = a
        self.w = wts.to(torch.bfloat16).double().tolist() if wts is not None else None
        eye = torch.eye(math.prod(n), dtype=torch.float64, device=dev)
        self.coarse = (eye - a * self.lv[-1][1](eye.view([-1] + n[::-1])).reshape(eye.shape)).T.contiguous()

    def resid(self, L, x, b):
        return (b - x) + self.a * self.lv[L][1](x)

    def smooth(self, L, x, b):
        for _ in range(2):
            r = self.resid(L, x, b)
            x = x + (_network(self.w, r)[1] if L == 0 and self.w is not None else 0.8 / self.lv[L][2] * r)
        return x

    def __call__(self, x, b, L=0):
        if L == len(self.lv) - 1:
            return torch.linalg.solve(self.coarse, b.reshape(-1)).view(b.shape)
        x = self.smooth(L, x, b)
        r = self.resid(L, x, b)
        for ax in range(r.dim()):
            m = r.shape[ax]
            r = 0.25 * r.narrow(ax, 0, m - 2) + 0.5 * r.narrow(ax, 1, m - 2) + 0.25 * r.narrow(ax, 2, m - 2)
            r = r.index_select(ax, torch.arange(0, m - 2, 2, device=r.device))
        e = self(torch.zeros_like(r), r, L + 1)
        for ax in range(e.dim()):
            m = e.shape[ax]
            p = torch.zeros([s if q != ax else 2 * m + 1 for q, s in enumerate(e.shape)], dtype=e.dtype, device=e.device)
            even = torch.arange(0, 2 * m, 2, device=e.device)
            p.index_add_(ax, even + 1, e)
            p.index_add_(ax, even, e, alpha=0.5)
            p.index_add_(ax, even + 2, e, alpha=0.5)
            e = p
        return self.smooth(L, x + e, b)


def _taps():
    return [(z, y, x) for z in (-1, 0, 1) for y in (-1, 0, 1) for x in (-1, 0, 1)]


def _shift(up, o):
    nz, ny, nx = (s - 2 for s in up.shape)
    return up[1 + o[0]:1 + o[0] + nz, 1 + o[1]:1 + o[1] + ny, 1 + o[2]:1 + o[2] + nx]


def _network(w, r):
    """Hidden fields and output of the two linear 3x3x3 layers (zero outside the box)."""
    pad = torch.nn.functional.pad
    rp = pad(r, (1,) * 6)
    y, hidden = torch.zeros_like(r), []
    for c in range(8):
        hc = torch.zeros_like(r)
        for t, o in enumerate(_taps()):
            hc.add_(_shift(rp, o), alpha=w[c * 27 + t])
        hp = pad(hc, (1,) * 6)
        for t, o in enumerate(_taps()):
            y.add_(_shift(hp, o), alpha=w[216 + c * 27 + t])
        hidden.append(hc)
    return hidden, y


def _exact_implicit(case, v):
    h = [l / (m + 1) for l, m in zip(case["length"], case["n"])]
    a, w = _half_dt2(case["omega"], case["spp"])
    plan = _plan(w, case["periods"], case["spp"])
    if case["rtol"] > 0.0:
        return _implicit_solved(case, v, h, a, plan)
    wts = _smoother_weights(case, 432, case["length"]) if case["learned"] else None
    cyc = _Cycle(case, h, a, v.device, wts)
    Nt, _, c = plan
    wm = v.double().view(case["n"][::-1])

    def solve(b):
        x = b
        for _ in range(case["cycles"]):
            x = cyc(x, b)
        return x

    w0 = solve(wm)
    acc = c[0] * wm + c[1] * w0
    for k in range(1, Nt):
        wm, w0 = w0, solve(2.0 * w0) - wm
        acc.add_(w0, alpha=c[k + 1])
    return acc.reshape(-1)


def _exact_smoother(case, state):
    n = case["n"][::-1]
    w = state["wts"].to(torch.bfloat16).double().tolist()
    r = state["r"].to(torch.bfloat16).double().view(n)
    gy = state["gy"].double().view(n)
    hidden, y = _network(w, r)
    pad = torch.nn.functional.pad
    rp, gp, grad = pad(r, (1,) * 6), pad(gy, (1,) * 6), torch.empty(432, dtype=torch.float64, device=r.device)
    for c in range(8):
        hp, gh = pad(hidden[c], (1,) * 6), torch.zeros_like(r)
        for t, o in enumerate(_taps()):
            grad[216 + c * 27 + t] = (gy * _shift(hp, o)).sum()
            gh.add_(_shift(gp, [-q for q in o]), alpha=w[216 + c * 27 + t])
        for t, o in enumerate(_taps()):
            grad[c * 27 + t] = (gh * _shift(rp, o)).sum()
    return {"y": y.reshape(-1), "grad": grad}


def _exact_eigs(case, start):
    n, dev = case["n"], start.device
    h = [l / (m + 1) for l, m in zip(case["length"], n)]
    lam2 = _symbol(n[0], h[0], case["order"], dev)[None, :] + _symbol(n[1], h[1], case["order"], dev)[:, None]
    lam = lam2.reshape(-1).sqrt()
    near = torch.argsort((lam - case["omega"]).abs())[:400]
    Nt, dt, c = _plan(case["omega"], _eigs_periods(case), _spp(case))
    lt = 2.0 / dt * torch.asin(0.5 * dt * lam[near])
    t = torch.arange(Nt + 1, dtype=torch.float64, device=dev) * dt
    beta = torch.cos(lt[:, None] * t[None, :]) @ torch.tensor(c, dtype=torch.float64, device=dev)
    top = near[torch.argsort(beta, descending=True)[:case["wanted"]]]
    ax = [torch.arange(1, m + 1, dtype=torch.float64, device=dev) * (math.pi / (m + 1)) for m in n]
    vecs = []
    for q in top.tolist():
        s = torch.sin((q // n[0] + 1) * ax[1])[:, None] * torch.sin((q % n[0] + 1) * ax[0])[None, :]
        s = (s / s.norm()).reshape(-1)
        vecs.append(s if float(s @ start[:s.numel()]) >= 0 else -s)
    return {"lam": lam[top].cpu().numpy(), "vecs": torch.stack(vecs)}


def exact(case, seed):
    case = _open(case)
    kind = case["kind"]
    if kind == "box":
        v = _uniform(math.prod(_active(case)) * case["nvec"], seed, _dtype(case["prec"]))
        return _exact_box(case, v)
    if kind == "batched":
        return [_exact_box(b, _uniform(math.prod(b["n"]), seed + 1000 * q, torch.float32))
                for q, b in enumerate(_boxes(case))]
    if kind == "mapped":
        return _exact_mapped(case, _uniform(math.prod(case["n"]) * case["nvec"], seed, _dtype(case["prec"])))
    if kind == "implicit":
        return _exact_implicit(case, _uniform(math.prod(case["n"]), seed, _dtype(case["prec"])))
    if kind == "smoother":
        n = math.prod(case["n"])
        return _exact_smoother(case, dict(wts=_smoother_weights(case, seed + 1, [1.0, 1.0, 1.0]),
                                          r=_uniform(n, seed, torch.float32),
                                          gy=_uniform(n, seed + 2, torch.float32)))
    return _exact_eigs(case, _uniform(math.prod(case["n"]) * case["block"], seed, torch.float64))
