"""lbm_step recorded by the caller into a CUDA graph: a replay reads the boundary arrays as
they are then, also on sides that held no values when the steps were recorded.  The replays
against the same calls made directly, bit for bit (the same kernels and arithmetic)."""
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


@pytest.mark.parametrize("prec", [0, 1])
@pytest.mark.parametrize("side", [2, 3])
def test_replay_reads_values_uploaded_after_the_capture(side, prec):
    nx, ny = 70, 24
    w = wl.channel(nx=nx, ny=ny, steps=0, Re=100.0 * ny / 256)
    rho0 = w["params"]["rho0"]
    q = 5e4 * (1.0 + 0.5 * np.sin(np.linspace(0, 6.0, nx)))
    moving = np.concatenate([np.full(nx, 1e-3), np.zeros(nx)])

    def solver(stream):
        s = lbm.Solver(w["params"], precision=prec, stream=stream.cuda_stream)
        for bc in w["bcs"]:
            s.set_bc(*bc)
        for wall in (2, 3):  # at rest, adiabatic: no values
            s.set_bc(wall, wl.BC_VELOCITY, None, rho0, wl.TBC_FLUX, None)
        s.init(**w["init"])
        s.step(1)
        return s

    st = torch.cuda.Stream()
    a, b = solver(st), solver(st)
    st.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=st):
        a.step(2)  # (advances the handle's counters as the first replay does its fields)
    for k in range(3):
        if k:
            for s in (a, b):
                s.set_bc(side, wl.BC_VELOCITY, moving * k, rho0, wl.TBC_FLUX, q * k)
        with torch.cuda.stream(st):
            graph.replay()
        b.step(2)
    st.synchronize()
    ma, mb = a.moments(), b.moments()
    for k in mb:
        assert np.array_equal(ma[k], mb[k]), k
    a.close()
    b.close()
