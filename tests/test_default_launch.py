"""The grid launch a solve takes by its size (nothing set by lbm_set_launch) against an
explicit 64 x 4 launch: bit for bit (the block shape does not enter the arithmetic) where
the same build runs, in FP32 to 4 x steps x 2^-24 of each field's magnitude (the
largest speed for both velocity components) where the size picks the build for more resident blocks.  Sizes on both sides of the rule's lines:
a single column of blocks, one wave of one-warp blocks and just above it, widths that
64- and 128-wide blocks do not divide, one row, and more rows than a grid dimension has
blocks of one row."""
import numpy as np
import pytest

from _helpers import run_gpu
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


def _fields(w, prec, steps, launch):
    s = lbm.Solver(w["params"], precision=prec)
    for bc in w["bcs"]:
        s.set_bc(*bc)
    if launch:
        s.set_launch(*launch)
    assert s.launch_config() == (0, 64, 4, 0)
    s.init(**(w.get("init") or {}))
    s.step(steps)
    m = s.moments(lbm.LBM_RHO | lbm.LBM_UX | lbm.LBM_UY | (lbm.LBM_T if w["params"]["thermal"] else 0))
    s.close()
    return m


@pytest.mark.parametrize("prec", [0, 1])
@pytest.mark.parametrize("nx,ny", [(33, 4), (2, 2), (608, 192), (608, 257), (1025, 152), (130, 1200)])
def test_default_launch_equals_nominal(nx, ny, prec):
    w = wl.channel(nx=nx, ny=ny, steps=0, Re=100.0 * ny / 256)
    a, b = _fields(w, prec, 9, None), _fields(w, prec, 9, (0, 64, 4))
    for k in a:
        assert np.array_equal(a[k], b[k]), k


def test_default_launch_large_fp32():
    """2400 x 520 nodes: two FP32 state buffers of 70 MB exceed L2, the build for more
    resident blocks runs."""
    steps = 9
    w = wl.channel(nx=2400, ny=520, steps=0, Re=100.0 * 520 / 256)
    a, b = _fields(w, 1, steps, None), _fields(w, 1, steps, (0, 64, 4))
    for k in a:
        scale = np.max(np.hypot(b["ux"], b["uy"])) if k in ("ux", "uy") else np.max(np.abs(b[k]))
        assert np.max(np.abs(a[k] - b[k])) <= 4 * steps * 2.0 ** -24 * scale, k


@pytest.mark.parametrize("nx,ny", [(40, 1), (1, 40), (4, 70000)])
def test_default_launch_thin_grids(nx, ny):
    """Rows beyond a grid dimension's 65535 blocks fall back to the nominal shape."""
    w = wl.poiseuille(nx=nx, ny=ny, steps=0)
    a, b = _fields(w, 0, 5, None), _fields(w, 0, 5, (0, 64, 4))
    for k in a:
        assert np.array_equal(a[k], b[k]), k
