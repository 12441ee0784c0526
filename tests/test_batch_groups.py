"""FP32 batches of more state than L2 holds, advanced group by group: every channel equals
the same channel stepped alone to 4 x steps x 2^-24 of each field's magnitude (the kernels
inline the same arithmetic in different contexts), over calls of fewer and more steps than
the rule's line, from either buffer, with channels that run as single solves (more than
16 MB of state), several that share a group, a group that the next channel overflows, and
boundary values that change between calls."""
import numpy as np
import pytest

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


SHAPES = [(33, 7), (1100, 700), (640, 300), (350, 350), (351, 349), (70, 24), (349, 352), (900, 512), (360, 333), (350, 340)]


@pytest.mark.parametrize("calls", [(57,), (1, 3, 4), (2, 5, 70), (4, 4, 1)])
@pytest.mark.parametrize("cfg", [None, (32, 8, 11)])
def test_groups_equal_one_by_one(calls, cfg):
    ws = [wl.channel(nx=nx, ny=ny, steps=0, Re=100.0 * ny / 256) for nx, ny in SHAPES]
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
        b.step(n)
        for s in solo:
            s.step(n)
    for k, s in enumerate(solo):
        a, r = b.channels[k].moments(), s.moments()
        for key in ("ux", "uy", "T", "rho"):
            scale = np.max(np.hypot(r["ux"], r["uy"])) if key in ("ux", "uy") else np.max(np.abs(r[key]))
            assert np.max(np.abs(a[key] - r[key])) <= 4 * sum(calls) * 2.0 ** -24 * scale, (k, key)
        assert b.channels[k].steps == sum(calls)
        s.close()
    b.close()


def test_one_channel_batch_equals_solo():
    """A batch of one channel, which runs as a single solve."""
    w = wl.channel(nx=640, ny=300, steps=0, Re=100.0 * 300 / 256)
    b, s = lbm.Batch([w["params"]], precision=1), lbm.Solver(w["params"], precision=1)
    for one in (b.channels[0], s):
        one.apply_workload(w)
    b.step(70)
    s.step(70)
    a, r = b.channels[0].moments(), s.moments()
    for key in ("ux", "uy", "T", "rho"):
        scale = np.max(np.hypot(r["ux"], r["uy"])) if key in ("ux", "uy") else np.max(np.abs(r[key]))
        assert np.max(np.abs(a[key] - r[key])) <= 4 * 70 * 2.0 ** -24 * scale, key
    s.close()
    b.close()
