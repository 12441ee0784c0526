"""LBM_LAUNCH_AUTO puts the launch by grid size back after an explicit one, after the TMA-staged
one and after the autotuner.  300 x 200 nodes in FP32 run one-warp blocks by size, about twice
as fast as the nominal 64 x 4 blocks (4 to 5 us against 9 us a step), so the time tells them
apart; the fields are those of a solve on which nothing was set, bit for bit."""
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


def _time(s, st):
    out = []
    s.step(129)
    for _ in range(5):
        e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        torch.cuda.synchronize()
        e0.record(st)
        s.step(256)
        e1.record(st)
        torch.cuda.synchronize()
        out.append(e0.elapsed_time(e1))
    return statistics.median(out)


def test_auto_returns_to_the_rule():
    w = wl.channel(nx=300, ny=200, steps=0, Re=100.0 * 200 / 256)
    st = torch.cuda.Stream()
    a, b = (lbm.Solver(w["params"], precision=1, stream=st.cuda_stream) for _ in range(2))
    for s in (a, b):
        s.apply_workload(w)
    t_default = _time(a, st)
    b.set_launch(lbm.LBM_LAUNCH_GRID, 64, 4)
    t_nominal = _time(b, st)
    assert t_nominal > 1.3 * t_default
    for change in (lambda: None, lambda: b.set_launch(lbm.LBM_LAUNCH_TMA, 4, 2, 1), b.autotune):
        change()
        b.set_launch(lbm.LBM_LAUNCH_AUTO)
        assert b.launch_config() == (lbm.LBM_LAUNCH_GRID, 64, 4, 0)
        assert _time(b, st) < 1.1 * t_default
    for s in (a, b):
        s.apply_workload(w)
        s.step(70)
    ma, mb = a.moments(), b.moments()
    for k in ma:
        assert np.array_equal(ma[k], mb[k]), k
    for bad in [(3, 64, 0, 0), (3, 0, 4, 0), (3, 0, 0, 1), (4, 0, 0, 0)]:
        with pytest.raises(lbm.LbmError):
            a.set_launch(*bad)
    a.close()
    b.close()
