"""Two-phase steps on grids of at most 16 columns (one-warp blocks of whole rows) against the
oracle: one column, columns that divide a warp and that do not, walls in x, in y, on all
sides and none, with and without a force field; 41 rows, so that the last block is short.
FP64, 1e-12 relative max-norm on phi, u and the post-collision h, z over 20 steps (the bounds of
test_parity_mp.py).

FP32: the same kernels on a slab that is uniform along x, whose columns must all stay equal
bit for bit, on every width: what a block's rows, its images beside them and its halo rows
hold shows in them."""
import numpy as np
import pytest

from _helpers import rel_max, run_gpu, run_oracle
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


def _slab(nx, ny, walls, wave=1.0):
    """A liquid slab with wavy faces, moving."""
    fl = dict(wl.AIR_WATER_25C, sigma=1e-4)
    H = 0.5e-3
    dx = H / ny
    dt = 0.1 * dx * dx / (3.0 * fl["nu_l"])
    w = wl.layered_poiseuille(fl, H=H, dx=dx, dt=dt, nx=nx, W=4 * dx, steps=20)
    x = np.arange(nx)[None, :] * (2 * np.pi / nx)
    y = (np.arange(ny) + 0.5)[:, None]
    d = np.abs(y - 0.5 * ny + 1.5 * wave * np.cos(x + 0.4)) - 0.25 * ny
    u = 0.02 * dx / dt
    sy = np.sin(2 * np.pi * y / ny)
    w["init"] = dict(a=0.5 - 0.5 * np.tanh(d / 2.0), ux=u * (1.0 + 0.3 * wave * sy * np.cos(x)), uy=0.5 * u * sy + 0.0 * x, b=None)
    w["bcs"] = [(s, wl.BC_WALL, None, w["params"]["rho_l"], wl.TBC_NONE, None) for s in range(4) if "xxyy"[s] in walls]
    return w


@pytest.mark.parametrize("force", [False, True])
@pytest.mark.parametrize("walls", ["", "x", "y", "xy"])
@pytest.mark.parametrize("nx", [1, 3, 10, 16])
def test_narrow(nx, walls, force):
    ny = 41
    w = _slab(nx, ny, walls)
    kw = {}
    if force:
        kw["force"] = 500.0 * np.random.default_rng(nx).standard_normal((2, ny, nx))
    o, s = run_oracle(w, **kw), run_gpu(w, 0, **kw)
    mo, mg = o.moments(), s.moments()
    sp = np.hypot(mo["ux"], mo["uy"])
    assert np.isfinite(sp).all() and sp.max() > 0
    assert rel_max(mg["phi"], mo["phi"]) < 1e-12
    assert rel_max(mg["ux"], mo["ux"], sp) < 1e-12 and rel_max(mg["uy"], mo["uy"], sp) < 1e-12
    st = s.state_arrays()
    assert rel_max(st["h"], o.dist("h", post=True)) < 1e-12
    assert rel_max(st["z"], o.dist("z", post=True)) < 1e-12
    s.close()


@pytest.mark.parametrize("force", [False, True])
@pytest.mark.parametrize("walls", ["", "y"])
def test_narrow_fp32_columns(walls, force):
    ny, ref = 41, None
    profile = 500.0 * np.random.default_rng(2).standard_normal((2, ny, 1))
    for nx in (1, 2, 3, 10, 16):
        w = _slab(nx, ny, walls, wave=0.0)
        s = run_gpu(w, 1, **(dict(force=np.repeat(profile, nx, axis=2)) if force else {}))
        st = np.concatenate(list(s.state_arrays().values()))
        s.close()
        ref = st[:, :, :1] if ref is None else ref
        assert np.isfinite(st).all() and np.array_equal(st, np.broadcast_to(ref, st.shape)), nx
