"""FP32 gradients against the FP64 form over 2000 steps.  Each step rounds a variable about four
times, by 2^-25 / sqrt(3) rms of its value; over N steps of independent roundings that is
sqrt(4 N / 3) 2^-25 (1.5e-6 at N = 2000), and the bound is three times that: 4.6e-6 relative L2
on the gradients of the heat source and of the wall flux, and of its value on that of nu.  (With
a temperature whose source is rounded the same way each step the first is 7e-6 off.)"""
import numpy as np
import pytest

from _helpers import rel_l2
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


@pytest.mark.parametrize("nx,ny,seed,off", [(1024, 128, 5, 0.01), (703, 109, 53, 0.04)])
def test_gradients(nx, ny, seed, off):
    steps, out = 2000, []
    w = wl.adjoint_channel(nx=nx, ny=ny, Re=50.0 * ny / 128)
    w["q3"] = wl.smooth_source(nx, ny, seed=seed)
    target = np.full(ny, w["T_in"]) + off * np.sin(np.pi * (np.arange(ny) + 0.5) / ny)
    for prec in (1, 0):
        s = lbm.Solver(w["params"], precision=prec)
        for bc in w["bcs"]:
            s.set_bc(*bc)
        s.set_source(w["q3"], None)
        s.init(**w["init"])
        out.append(lbm.lbm_adjoint(s.h, steps, 100, target, nx, ny))
        s.close()
    (_, g3, gw, gn), (_, r3, rw, rn) = out
    got = dict(q3=rel_l2(g3, r3), qwall=rel_l2(gw, rw), nu=abs(gn - rn) / abs(rn))
    assert max(got.values()) < 3 * np.sqrt(4 * steps / 3) * 2.0 ** -25, got
