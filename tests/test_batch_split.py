"""FP32 batches in which some channels take a call's steps as single solves and the others share
launches: every channel against the same channel stepped alone, to 4 x steps x 2^-24 of each
field's magnitude, over calls below and above the graph's 64 steps, from either buffer, with
boundary values, launches and so the split changing between calls; and the times of batches of
channels that gain nothing from it against the launch over all (calls of three steps)."""
import math
import statistics

import numpy as np
import pytest

from paper_2302_04120_gb300 import workloads as wl

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
lbm = pytest.importorskip("paper_2302_04120_gb300.lbm")


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2302_04120_gb300 import build
    build.build()


def _w(nx, ny):
    return wl.channel(nx=nx, ny=ny, steps=0, Re=100.0 * ny / 256)


def _same(a, r, steps, tag):
    for key in ("ux", "uy", "T", "rho"):
        scale = np.max(np.hypot(r["ux"], r["uy"])) if key in ("ux", "uy") else np.max(np.abs(r[key]))
        assert np.max(np.abs(a[key] - r[key])) <= 4 * steps * 2.0 ** -24 * scale, (tag, key)


# 88, 59, 67 MB: single solves in every call; 39 MB: in long ones; the others share launches
SHAPES = [(33, 7), (1100, 700), (351, 349), (1000, 512), (70, 24), (1060, 550), (800, 440), (350, 340)]


@pytest.mark.parametrize("calls", [(57,), (1, 3, 4), (2, 5, 70), (4, 64, 1)])
@pytest.mark.parametrize("cfg", [None, (32, 8, 11)])
def test_split_equals_one_by_one(calls, cfg):
    ws = [_w(nx, ny) for nx, ny in SHAPES]
    b = lbm.Batch([w["params"] for w in ws], precision=1)
    if cfg:
        b.config(*cfg)
    solo = [lbm.Solver(w["params"], precision=1) for w in ws]
    for a, s, w in zip(b.channels, solo, ws):
        for one in (a, s):
            one.apply_workload(w)
    for c, n in enumerate(calls):
        if c == 1:
            for one, w in zip(b.channels + solo, ws + ws):
                q = w["qflux"] * (1.0 + 0.5 * np.sin(np.linspace(0, 6.0, w["params"]["nx"])))
                one.set_bc(2, wl.BC_WALL, None, w["params"]["rho0"], wl.TBC_FLUX, q)
            b.channels[3].set_launch(lbm.LBM_LAUNCH_TMA, 4, 2, 1)  # joins the shared launches
            b.channels[5].set_launch(lbm.LBM_LAUNCH_GRID, 32, 8)
        if c == 2:
            b.channels[3].set_launch(lbm.LBM_LAUNCH_GRID, 64, 1)
        b.step(n)
        for s in solo:
            s.step(n)
    for k, s in enumerate(solo):
        _same(b.channels[k].moments(), s.moments(), sum(calls), k)
        assert b.channels[k].steps == sum(calls)
        s.close()
    b.close()


def test_tall_channel_with_a_launch_of_too_many_rows():
    """A channel whose own launch has more rows of blocks than a grid can have (lbm_step refuses
    it) advances in the batch, whose launches do not use it."""
    steps = 9
    ws = [_w(8, 70000), _w(1100, 700), _w(33, 7)]
    b = lbm.Batch([w["params"] for w in ws], precision=1)
    s = lbm.Solver(ws[0]["params"], precision=1)
    for one, w in zip(b.channels + [s], ws + [ws[0]]):
        one.apply_workload(w)
    b.channels[0].set_launch(lbm.LBM_LAUNCH_GRID, 32, 1)
    b.step(5)
    b.step(4)
    s.step(steps)
    _same(b.channels[0].moments(), s.moments(), steps, "tall")
    assert [c.steps for c in b.channels] == [steps] * 3
    s.close()
    b.close()


def test_captured_call_after_a_launch_change():
    """A channel's launch set just before the caller captures a call: the capture holds, and its
    replay advances every channel as the call itself does."""
    ws = [_w(nx, ny) for nx, ny in [(1100, 700), (1000, 512), (33, 7), (1060, 550)]]
    st = torch.cuda.Stream()
    out = []
    for captured in (True, False):
        b = lbm.Batch([w["params"] for w in ws], precision=1, stream=st.cuda_stream)
        for ch, w in zip(b.channels, ws):
            ch.apply_workload(w)
        b.step(7)
        b.step(4)  # (the tables are those of this call's buffers, which a capture cannot upload)
        st.synchronize()
        b.channels[1].set_launch(lbm.LBM_LAUNCH_TMA, 4, 2, 1)
        if captured:
            graph = torch.cuda.CUDAGraph()
            with torch.cuda.graph(graph, stream=st):
                b.step(6)
            with torch.cuda.stream(st):
                graph.replay()
        else:
            b.step(6)
        st.synchronize()
        out.append([ch.moments() for ch in b.channels])
        b.close()
    for k, (a, r) in enumerate(zip(*out)):
        _same(a, r, 17, k)


def _shape(mb, k):
    nodes = mb * 1e6 / 112
    nx = int(round(math.sqrt(4 * nodes))) + k % 5
    return nx, max(8, int(round(nodes / nx)))


@pytest.mark.parametrize("sizes", [[10] * 8, [5] * 48, [16] * 24, [30] * 8, [180] * 4, [60, 30, 20, 10, 5, 2, 1]])
def test_no_slower_than_one_launch_over_all(sizes):
    """Sizes in MB of both buffers.  The bound leaves 10 % for the spread of the medians."""
    st = torch.cuda.Stream()
    shapes = [_shape(mb, k) for k, mb in enumerate(sizes)]
    b = lbm.Batch([_w(*x)["params"] for x in shapes], precision=1, stream=st.cuda_stream)
    for ch, x in zip(b.channels, shapes):
        for bc in _w(*x)["bcs"]:
            ch.set_bc(*bc)
        ch.init()
    b.step(3)
    t = {48: [], 3: []}
    for _ in range(5):
        for n in t:
            e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            b.step(n)
            torch.cuda.synchronize()
            e0.record(st)
            for _ in range(96 // n):
                b.step(n)
            e1.record(st)
            torch.cuda.synchronize()
            t[n].append(e0.elapsed_time(e1))
    b.close()
    assert statistics.median(t[48]) <= 1.1 * statistics.median(t[3]), t
