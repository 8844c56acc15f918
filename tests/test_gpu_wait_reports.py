"""Wave-solves whose kernels wait (one cooperative launch a solve, staged copies) from two threads on streams of their
own, and who hears of a wait that gave up: the grid it happened on and the thread that launched it, nobody else."""
import threading

import numpy as np
import pytest
import torch

import ew_inputs

pytestmark = pytest.mark.gpu
EW_ETIMEOUT = 6


@pytest.fixture(scope="module")
def ew():
    import __graft_entry__
    __graft_entry__.build()
    import paper_2507_18282_gb300 as ew
    return ew


def _problem(ew, n, order, nvec, mapped=False):
    if mapped:
        r, s = np.meshgrid(np.linspace(0, 1, n[0] + 2), np.linspace(0, 1, n[1] + 2))
        g = ew.ew_grid_create_mapped(n, np.stack([r + 0.05 * np.sin(6 * s) * r * (1 - r), s], -1), "fp32")
    else:
        g = ew.ew_grid_create(2, n, (1.0, 0.9), order=order, prec="fp32")
    v = torch.tensor(ew_inputs.uniform_pm1(41, g.size * nvec), dtype=torch.float32, device="cuda")
    return g, ew.filter_params(25.0), v


def test_two_threads_on_two_streams(ew):
    shapes = [((300, 250), 4, 2, False), ((517, 389), 2, 1, False), ((1301, 700), 4, 2, False), ((401, 300), 2, 2, True)]
    probs = [_problem(ew, *s) for s in shapes] + [_problem(ew, *s) for s in shapes]
    refs = []
    for (g, p, v), s in zip(probs, shapes + shapes):
        refs.append(torch.empty_like(v))
        ew.ew_filter_apply(g, p, v, refs[-1], nvec=s[2])
    torch.cuda.synchronize()
    errors = []

    def work(k):
        try:
            st = torch.cuda.Stream()
            mine = list(range(k * len(shapes), (k + 1) * len(shapes)))
            if k:
                mine.reverse()
            with torch.cuda.stream(st):
                for _ in range(6):
                    outs = {}
                    for q in mine:
                        g, p, v = probs[q]
                        outs[q] = torch.full_like(v, float("nan"))
                        ew.ew_filter_apply(g, p, v, outs[q], nvec=shapes[q % len(shapes)][2])
                    for q in mine:
                        ew.ew_rayleigh(probs[q][0], outs[q], nvec=1)
                        assert torch.equal(outs[q], refs[q]), shapes[q % len(shapes)]
        except BaseException as e:  # noqa: BLE001 (reported below)
            errors.append(e)

    ts = [threading.Thread(target=work, args=(k,)) for k in range(2)]
    for t in ts:
        t.start()
    for t in ts:
        t.join()
    assert not errors, errors
    for g, _, _ in probs:
        g.close()


def test_report_reaches_its_grid_and_thread(ew, monkeypatch):
    a, pa, va = _problem(ew, (300, 250), 4, 1)
    b, pb, vb = _problem(ew, (310, 260), 4, 1)
    wa, wb = torch.empty_like(va), torch.empty_like(vb)
    seen = {}

    def stalled():
        monkeypatch.setenv("EW_TEST_RB2D_STALL", "1")
        ew.ew_filter_apply(a, pa, va, wa)
        monkeypatch.delenv("EW_TEST_RB2D_STALL")
        torch.cuda.synchronize()

    def status(name, grid, x):
        try:
            ew.ew_rayleigh(grid, x)
            seen[name] = 0
        except ew.EWError as e:
            seen[name] = e.status

    def run(f, *args):
        t = threading.Thread(target=f, args=args)
        t.start()
        t.join()

    # launched here: another thread's check on another grid neither hears of it nor takes it away
    stalled()
    run(status, "other thread, other grid", b, vb)
    status("same thread, other grid", b, vb)
    status("told once", a, va)
    # launched by a thread that is gone: the grid still reports it, once, to whoever asks
    run(stalled)
    status("this thread, other grid", b, vb)
    status("this thread, its grid", a, va)
    status("told once more", a, va)
    assert seen == {"other thread, other grid": 0, "same thread, other grid": EW_ETIMEOUT, "told once": 0,
                    "this thread, other grid": 0, "this thread, its grid": EW_ETIMEOUT, "told once more": 0}
    # the handle may go before its thread looks
    stalled()
    a.close()
    status("after the handle is gone", b, vb)
    assert seen["after the handle is gone"] == EW_ETIMEOUT
    ew.ew_filter_apply(b, pb, vb, wb)
    status("clean", b, vb)
    assert seen["clean"] == 0
    b.close()
