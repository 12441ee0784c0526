"""MRT with the free rates of e and eps away from one (omega_e_dt, omega_eps_dt): the step
and the adjoint against the oracle, without and with forces.  The bounds of the unit rates
(test_parity_sp.py, test_adjoint.py): FP64 1e-12 relative max-norm on u, T - T_in and the
post-collision deviations against the long-double oracle, FP32 1e-5 relative L2; gradients
1e-8 relative max-norm, FP32 1e-3."""
import functools

import numpy as np
import pytest

from _helpers import W5, W9, deviations, rel_l2, rel_max, run_gpu, run_oracle
from paper_2302_04120_gb300 import workloads as wl

pytestmark = pytest.mark.gpu

lbm = pytest.importorskip("paper_2302_04120_gb300.lbm")
RATES = [(1.3, 1.0), (1.0, 0.8), (0.7, 1.6)]


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2302_04120_gb300 import build
    build.build()


def _channel(nx, ny, steps, rates):
    w = wl.channel(nx=nx, ny=ny, steps=steps, Re=100 * ny / 256)
    w["params"].update(omega_e_dt=rates[0], omega_eps_dt=rates[1])
    return w


def _force(nx, ny):
    return 50.0 * np.random.default_rng(11).standard_normal((2, ny, nx))


@pytest.mark.parametrize("prec", [0, 1])
@pytest.mark.parametrize("forced", [False, True])
@pytest.mark.parametrize("rates", RATES)
def test_step(rates, forced, prec):
    nx, ny = 70, 36
    w = _channel(nx, ny, 150, rates)
    kw = dict(force=_force(nx, ny)) if forced else {}
    o, s = run_oracle(w, extended=prec == 0, **kw), run_gpu(w, prec, **kw)
    mo, mg = o.moments(), s.moments()
    sp, T_in = np.hypot(mo["ux"], mo["uy"]), w["T_in"]
    norm, tol = (rel_max, 1e-12) if prec == 0 else (rel_l2, 1e-5)
    assert norm(mg["ux"], mo["ux"], sp) < tol and norm(mg["uy"], mo["uy"], sp) < tol
    assert norm(mg["T"] - T_in, mo["T"] - T_in) < tol
    if prec == 0:
        st, p = s.state_arrays(deviations=True), w["params"]
        assert rel_max(st["f"], deviations(o.dist("f", post=True), W9, p["rho0"])) < tol
        assert rel_max(st["g"], deviations(o.dist("g", post=True), W5, p.get("T0", 300.0))) < tol
    s.close()


def _gradient_setup(rates, forced):
    nx, ny, steps = 32, 10, 80
    w = _channel(nx, ny, steps, rates)
    if forced:
        w["params"]["Fb"] = (40.0, -25.0)
    w["q3"] = wl.smooth_source(nx, ny, seed=5, sigma_cells=2.0, scale=1e8)
    # 1 K off, so that FP32's rounding of T does not decide the seed of the reverse sweep
    target = run_oracle(w).moments()["T"][:, -1] + 1.0 + 0.5 * np.sin(np.pi * (np.arange(ny) + 0.5) / ny)
    return w, steps, target


@functools.lru_cache(maxsize=None)
def _reference(rates, forced):
    import oracle
    w, steps, target = _gradient_setup(rates, forced)
    return oracle.outlet_loss_gradient(w, steps, target)


@pytest.mark.parametrize("prec,tol", [(0, 1e-8), (1, 1e-3)])
@pytest.mark.parametrize("forced", [False, True])
@pytest.mark.parametrize("rates", RATES)
def test_adjoint(rates, forced, prec, tol):
    w, steps, target = _gradient_setup(rates, forced)
    s = lbm.Solver(w["params"], precision=prec)
    for bc in w["bcs"]:
        s.set_bc(*bc)
    s.set_source(w["q3"], None)
    s.init(**w["init"])
    loss, g3, gw, gnu = lbm.lbm_adjoint(s.h, steps, 25, target, s.nx, s.ny)
    s.close()
    L, r3, rw, rnu = _reference(rates, forced)
    assert abs(loss - L) <= (1e-7 if prec == 0 else 2e-3) * L
    assert rel_max(g3, r3) < tol and rel_max(gw, rw) < tol and abs(gnu - rnu) <= tol * abs(rnu)
