"""FP32 over thousands of steps: T - T_in of the thermal MRT forms, with a heat source whose
share of one step is about a unit in the last place of sum g, and without, against the FP64
form of the same run.  Bound: the contract of the FP32 form, 1e-5 relative L2 on T - T_in and
on u (a source rounded the same way each step leaves it after a few hundred steps).

And a weak source over 10000 steps: the roundings are those of the run without it, so its
error is held to three times that run's."""
import numpy as np
import pytest

from _helpers import rel_l2, run_gpu
from paper_2302_04120_gb300 import workloads as wl

pytestmark = pytest.mark.gpu

lbm = pytest.importorskip("paper_2302_04120_gb300.lbm")


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2302_04120_gb300 import build
    build.build()


def _waves(nx, ny, phase):
    x, y = np.arange(nx)[None, :] * (2 * np.pi / nx), np.arange(ny)[:, None] * (2 * np.pi / ny)
    return np.cos(2 * x + phase) * np.sin(y + 0.3) + 0.7 * np.sin(x - phase) * np.cos(2 * y + phase)


def _error(w, steps, T_in):
    a, b = run_gpu(w, 1, steps=steps), run_gpu(w, 0, steps=steps)
    ma, mb = a.moments(), b.moments()
    a.close()
    b.close()
    sp = np.hypot(mb["ux"], mb["uy"])
    return dict(T=rel_l2(ma["T"], mb["T"], mb["T"] - T_in), ux=rel_l2(ma["ux"], mb["ux"], sp), uy=rel_l2(ma["uy"], mb["uy"], sp))


def _problem(kind, q, nx, ny):
    if kind == "d2q9":
        w = wl.heated_channel(nx=nx, ny=ny, steps=0, flow_op=1)
        T_in = w["params"]["T0"]
    else:
        w = wl.channel(nx=nx, ny=ny, steps=0, Re=100 * ny / 256, flow_op=int(kind == "d2q5"))
        T_in = w["T_in"]
    init = dict(w["init"])
    init["b"] = (T_in if init.get("b") is None else np.asarray(init["b"])) + 2.0 * _waves(nx, ny, 0.5) + np.zeros((ny, nx))
    w["init"] = init
    if q:
        w["q3"] = q * _waves(nx, ny, 1.1)
    return w, T_in


@pytest.mark.parametrize("q", [0.0, 1e6, 1e8])
@pytest.mark.parametrize("kind", ["d2q5", "d2q5_bgk_flow", "d2q9"])
def test_temperature_keeps_its_source(kind, q):
    w, T_in = _problem(kind, q, *((500, 50) if kind == "d2q9" else (400, 100)))
    got = _error(w, 4000, T_in)
    assert max(got.values()) < 1e-5, got


@pytest.mark.parametrize("kind,nx,ny", [("d2q5", 1024, 128), ("d2q9", 700, 96)])
def test_weak_source_adds_no_drift(kind, nx, ny):
    e = []
    for q in (0.0, 1e5):
        w, T_in = _problem(kind, q, nx, ny)
        e.append(_error(w, 10000, T_in)["T"])
    assert e[1] < 3 * e[0], e
