"""Performance cases: what a user of the solver has it do, through its public calls.

Every pass is a run from given initial fields: lbm_init_fields with device arrays,
lbm_step(n), and the macroscopic fields read back into device arrays (lbm_moments), as
a user's program would do for a run of n steps; the control case steps once between
boundary uploads and an integrals read, and the adjoint case is one lbm_adjoint call.
FP32 solves hand their fields on in FP32, the precision they were computed in.

``exact`` solves the same inputs in float64 with plain torch: collide with explicit
moment matrices, then push; the adjoint's gradients come from autograd.
"""
import math

import numpy as np
import torch

from paper_2302_04120_gb300 import lbm

# Fluids: water of the forced-convection channel, water at 301 K (heated channel), air
# at 333.5 K (cavity), and the two-phase systems.
WATER = dict(rho0=1000.0, cp=4180.0, k=0.6)
ALPHA = WATER["k"] / (WATER["rho0"] * WATER["cp"])
WATER_301K = dict(rho0=996.279, nu=8.382e-7, k=0.611, cp=4180.333)
AIR_333K = dict(rho0=1.059, cp=1008.045, k=0.029, nu=1.90e-5)
TWO_PHASE = {
    "air_water": dict(rho_g=1.184, rho_l=997.048, nu_g=155.770e-7, nu_l=8.927e-7, sigma=0.072),
    "sat_water_100C": dict(rho_g=0.598, rho_l=958.349, nu_g=204.493e-7, nu_l=2.938e-7, sigma=0.059),
    "sat_water_80C": dict(rho_g=0.294, rho_l=971.766, nu_g=392.919e-7, nu_l=3.643e-7, sigma=0.063),
    "sat_water_25C": dict(rho_g=0.023, rho_l=997.003, nu_g=4204.120e-7, nu_l=8.927e-7, sigma=0.072),
}
BGK, MRT = lbm.LBM_BGK, lbm.LBM_MRT
OPS = {"bgk": BGK, "mrt": MRT}


# ---------------------------------------------------------------------------
# The cases
# ---------------------------------------------------------------------------
def listed():
    return [
        # The isothermal Poiseuille channel of the paper's first workload: 2112 nodes, so a
        # run is launches and latency.
        dict(name="poiseuille_64x33_f64", kind="poiseuille", nx=64, ny=33, op="bgk", prec="f64", steps=400),
        # The headline forced-convection channel, in the form most runs take (FP32).
        dict(name="channel_2048x256_f32", kind="channel", nx=2048, ny=256, op="mrt", top="mrt", prec="f32", steps=200),
        # The same channel in FP64, the form the validation runs take.
        dict(name="channel_2048x256_f64", kind="channel", nx=2048, ny=256, op="mrt", top="mrt", prec="f64", steps=24),
        # The roofline-size channel: 3.8 GB of state, far beyond L2.
        dict(name="channel_8192x4096_f32", kind="channel", nx=8192, ny=4096, op="mrt", top="mrt", prec="f32", steps=80),
        # A control loop around the headline channel: both wall-flux profiles uploaded from
        # the host, one step, the integrals read back and the temperature field handed on.
        dict(name="control_2048x256_f32", kind="control", nx=2048, ny=256, op="mrt", top="mrt", prec="f32", steps=1),
        # The paper's heated half channel, case 1 (D2Q9 BGK flow, D2Q9 MRT thermal lattice,
        # symmetry top, oscillating wall flux).
        dict(name="heated_2000x50_f32", kind="heated", nx=2000, ny=50, op="bgk", top="mrt", prec="f32", steps=200),
        # The static-bubble workload (conservative Allen-Cahn + pressure LBE) at its size.
        dict(name="bubble_512_f32", kind="bubble", nx=512, ny=512, fluid="sat_water_25C", op="mrt", prec="f32", steps=100),
        # The same model on the largest two-phase grid of the benchmark (2.1 GB of state).
        dict(name="bubble_4096_f32", kind="bubble", nx=4096, ny=4096, fluid="air_water", op="mrt", prec="f32", steps=80),
        # Layered two-phase flow between walls: the paper's 10 x 400 grid, FP64 (the form its
        # runs of tens of millions of steps take).
        dict(name="layered_10x400_f64", kind="layered", nx=10, ny=400, fluid="sat_water_100C", op="mrt", prec="f64",
             steps=200),
        # Many independent channels of uneven size in one launch per step.
        dict(name="batch_48_f32", kind="batch", count=48, spec=4, prec="f32", steps=48),
        # The gradient workload (heat source per cell, wall flux, viscosity), both forms.
        dict(name="adjoint_1024x128_f64", kind="adjoint", nx=1024, ny=128, every=20, prec="f64", steps=100),
        dict(name="adjoint_1024x128_f32", kind="adjoint", nx=1024, ny=128, every=50, prec="f32", steps=200),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _steps(rng, nodes, budget, most):
    """As many steps as a node budget allows, at most `most`, odd and even ones."""
    n = max(3, min(most, int(budget / nodes)))
    return max(3, n - rng.randrange(0, max(1, n // 4) + 1))


def draw(rng):
    kind = rng.choice(["poiseuille", "channel", "channel", "control", "heated", "cavity", "bubble", "layered", "batch",
                       "adjoint"])
    prec = rng.choice(["f32", "f32", "f64"])
    slow = 12.0 if prec == "f64" else 1.0
    op, top = rng.choice(["bgk", "mrt"]), rng.choice(["bgk", "mrt"])
    if kind == "poiseuille":
        nx, ny = _log(rng, 32, 4096), _log(rng, 9, 2048)
        return dict(kind=kind, nx=nx, ny=ny, op=op, prec=prec, steps=_steps(rng, nx * ny, 1.2e9 / slow, 400 if prec == "f64" else 120))
    if kind == "channel":
        nx, ny = _log(rng, 64, 6000), _log(rng, 16, 3000)
        return dict(kind=kind, nx=nx, ny=ny, op=op, top=top, prec=prec, steps=_steps(rng, nx * ny, 1.2e9 / slow, 300))
    if kind == "control":
        return dict(kind=kind, nx=_log(rng, 64, 4096), ny=_log(rng, 16, 512), op="mrt", top=top, prec=prec, steps=1)
    if kind == "heated":
        nx, ny = _log(rng, 100, 4000), _log(rng, 20, 200)
        return dict(kind=kind, nx=nx, ny=ny, op=op, top=top, prec=prec, steps=_steps(rng, nx * ny, 1e8 / slow, 300))
    if kind == "cavity":
        n = _log(rng, 33, 600)
        return dict(kind=kind, nx=n, ny=n, op=op, top=top, prec=prec, steps=_steps(rng, n * n, 1e8 / slow, 300))
    fluid = rng.choice(sorted(TWO_PHASE))
    if kind == "bubble":
        lo = 160 if prec == "f64" else 320
        nx, ny = _log(rng, lo, 2500), _log(rng, lo, 2500)
        return dict(kind=kind, nx=nx, ny=ny, fluid=fluid, op="mrt", prec=prec, steps=_steps(rng, nx * ny, 2e8 / slow, 60))
    if kind == "layered":
        # (BGK z is stable at the air-water density ratio only)
        op = op if fluid == "air_water" else "mrt"
        return dict(kind=kind, nx=_log(rng, 2, 64), ny=rng.choice([100, 200, 400]), fluid=fluid, op=op, prec="f64",
                    steps=rng.randrange(60, 201))
    if kind == "batch":
        return dict(kind=kind, count=_log(rng, 4, 48), spec=rng.randrange(1 << 16), prec=prec,
                    steps=rng.randrange(16, 41) if prec == "f32" else rng.randrange(4, 9))
    nx, ny = _log(rng, 64, 1500), _log(rng, 16, 256)
    steps = _steps(rng, nx * ny, 4e7 / slow, 150)
    return dict(kind="adjoint", nx=nx, ny=ny, every=max(2, steps // rng.randrange(3, 9)), prec=prec, steps=steps)


# ---------------------------------------------------------------------------
# Inputs
# ---------------------------------------------------------------------------
def _smooth(gen, nx, ny, modes=4):
    """A smooth field of about unit size on the device: a few random periodic modes."""
    x = torch.arange(nx, dtype=torch.float64, device="cuda")[None, :] * (2 * math.pi / nx)
    y = torch.arange(ny, dtype=torch.float64, device="cuda")[:, None] * (2 * math.pi / ny)
    out = torch.zeros((ny, nx), dtype=torch.float64, device="cuda")
    for _ in range(modes):
        kx, ky = int(gen.integers(0, 5)), int(gen.integers(0, 4))
        ax, ay = x * kx + float(gen.uniform(0, 6.3)), y * ky + float(gen.uniform(0, 6.3))
        out += float(gen.uniform(-1, 1)) * (torch.cos(ax) * torch.sin(ay))
    return out


def _full(nx, ny, v):
    return torch.full((ny, nx), float(v), dtype=torch.float64, device="cuda")


def _parabola(ny, u_mean):
    s = (np.arange(ny) + 0.5) / ny
    return 6.0 * u_mean * (s - s * s)


def _single(case, nx, ny, dx, dt, fluid, nu, T0, thermal, **more):
    p = dict(nx=nx, ny=ny, dx=dx, dt=dt, flow=9, flow_op=OPS[case.get("op", "mrt")], thermal=thermal, phase=0,
             rho0=fluid["rho0"], nu=nu, T0=T0)
    if thermal:
        p.update(thermal_op=OPS[case.get("top", "mrt")], cp=fluid["cp"], k=fluid["k"])
    p.update(more)
    return p


def _channel(case, gen, nx, ny, dx=2.5e-6, dt=6.25e-7, u_m=None, nu=7.0 * ALPHA):
    """Developing forced convection: parabolic inlet, pressure outlet, heated walls; the
    inlet speed of the 2048 x 256 workload at every height."""
    u_m = 100.0 * 7.0 * ALPHA / (2 * 256 * 2.5e-6) if u_m is None else u_m
    T_in, rho0 = 300.0, WATER["rho0"]
    uin = _parabola(ny, u_m * float(gen.uniform(0.9, 1.1)))
    qw = [4e4 * (1.0 + 0.5 * np.sin(np.arange(nx) * (2 * math.pi * float(gen.uniform(1, 4)) / nx))) for _ in range(2)]
    bcs = [(0, lbm.LBM_BC_VELOCITY, np.concatenate([uin, np.zeros(ny)]), rho0, lbm.LBM_TBC_TEMP, np.full(ny, T_in)),
           (1, lbm.LBM_BC_PRESSURE, None, rho0, lbm.LBM_TBC_OUTFLOW, None),
           (2, lbm.LBM_BC_WALL, None, rho0, lbm.LBM_TBC_FLUX, qw[0]),
           (3, lbm.LBM_BC_WALL, None, rho0, lbm.LBM_TBC_FLUX, qw[1])]
    u = torch.from_numpy(uin).cuda()[:, None]
    init = dict(a=None, ux=u * (1.0 + 0.1 * _smooth(gen, nx, ny)), uy=0.2 * u * _smooth(gen, nx, ny),
                b=T_in + 2.0 * _smooth(gen, nx, ny))
    return dict(params=_single(case, nx, ny, dx, dt, WATER, nu, T_in, 5), bcs=bcs, init=init, q3=None)


def _problem(case, seed):
    """Parameters, boundaries (host arrays) and initial fields (device) of one solve."""
    kind, gen = case["kind"], np.random.default_rng([seed, 77])
    nx, ny = case.get("nx", 0), case.get("ny", 0)
    if kind in ("channel", "control"):
        return _channel(case, gen, nx, ny)
    if kind == "adjoint":
        w = _channel(dict(case, op="mrt", top="mrt"), gen, nx, ny)
        w["q3"] = 1e6 * _smooth(gen, nx, ny)
        w["target"] = 301.0 + np.sin(math.pi * (np.arange(ny) + 0.5) / ny)
        return w
    if kind == "poiseuille":
        dx, nu, rho0, u_max = 1e-3 / 32, 1e-6, 1000.0, 1e-3
        Fb = 8.0 * rho0 * nu * u_max / (33 * dx) ** 2
        u = torch.from_numpy(_parabola(ny, u_max * 2 / 3)).cuda()[:, None]
        bcs = [(s, lbm.LBM_BC_WALL, None, rho0, lbm.LBM_TBC_NONE, None) for s in (2, 3)]
        return dict(params=_single(case, nx, ny, dx, 9.765625e-5, dict(rho0=rho0), nu, 300.0, 0, Fb=(Fb, 0.0)), bcs=bcs,
                    init=dict(a=None, ux=u * (1.0 + 0.2 * _smooth(gen, nx, ny)), uy=0.2 * u * _smooth(gen, nx, ny), b=None),
                    q3=None)
    if kind == "heated":
        f, u_m, T_in = WATER_301K, 0.2, 300.0
        s = (np.arange(ny) + 0.5) / (2 * ny)
        uin = 6.0 * u_m * float(gen.uniform(0.9, 1.1)) * (s - s * s)
        Tin = T_in + 4e4 * 5e-4 / f["k"] * (-s ** 4 + 2 * s ** 3 - s + 0.243)
        x = (np.arange(nx) + 0.5) * 5e-6
        qw = 4e4 + 4e4 * np.sign(np.sin(2 * math.pi * x / 1e-3 + float(gen.uniform(0, 6))))
        bcs = [(0, lbm.LBM_BC_VELOCITY, np.concatenate([uin, np.zeros(ny)]), f["rho0"], lbm.LBM_TBC_TEMP, Tin),
               (1, lbm.LBM_BC_PRESSURE, None, f["rho0"], lbm.LBM_TBC_OUTFLOW, None),
               (2, lbm.LBM_BC_WALL, None, f["rho0"], lbm.LBM_TBC_FLUX, qw),
               (3, lbm.LBM_BC_SYMMETRY, None, f["rho0"], lbm.LBM_TBC_SYMMETRY, None)]
        u = torch.from_numpy(uin).cuda()[:, None]
        init = dict(a=None, ux=u * (1.0 + 0.1 * _smooth(gen, nx, ny)), uy=0.2 * u * _smooth(gen, nx, ny),
                    b=torch.from_numpy(Tin).cuda()[:, None] + _smooth(gen, nx, ny))
        return dict(params=_single(case, nx, ny, 5e-6, 2e-6, f, f["nu"], T_in, 9), bcs=bcs, init=init, q3=None)
    if kind == "cavity":
        f, T_h, T_c = AIR_333K, 373.15, 293.85
        p = _single(case, nx, ny, 2e-4, 2e-4, f, f["nu"], T_c, 5, gravity=(0.0, -9.81), beta_exp=3.004e-3, T_ref=333.5,
                    rho_ref=f["rho0"])
        W, r = lbm.LBM_BC_WALL, f["rho0"]
        bcs = [(0, W, None, r, lbm.LBM_TBC_TEMP, np.full(ny, T_h)), (1, W, None, r, lbm.LBM_TBC_TEMP, np.full(ny, T_c)),
               (2, W, None, r, lbm.LBM_TBC_FLUX, np.zeros(nx)), (3, W, None, r, lbm.LBM_TBC_FLUX, np.zeros(nx))]
        init = dict(a=None, ux=0.02 * _smooth(gen, nx, ny), uy=0.02 * _smooth(gen, nx, ny), b=333.5 + 15.0 * _smooth(gen, nx, ny))
        return dict(params=p, bcs=bcs, init=init, q3=None)
    fl = TWO_PHASE[case["fluid"]]
    p = dict(nx=nx, ny=ny, flow=9, flow_op=MRT, thermal=0, phase=5, z_op=OPS[case["op"]], rho0=fl["rho_l"], mobility=1e-5, **fl)
    if kind == "bubble":
        dx, c = 5e-6, 50.0
        R, W = min(nx, ny) / 8.0 * float(gen.uniform(0.9, 1.1)), 5.0
        x = torch.arange(nx, dtype=torch.float64, device="cuda")[None, :] - nx * float(gen.uniform(0.4, 0.6))
        y = torch.arange(ny, dtype=torch.float64, device="cuda")[:, None] - ny * float(gen.uniform(0.4, 0.6))
        phi = 0.5 + 0.5 * torch.tanh(2.0 * (torch.sqrt(x * x + y * y) - R) / W)
        p.update(dx=dx, dt=1e-7, W=W * dx)
        # a drifting bubble: a uniform velocity of about 2 % of c
        init = dict(a=phi, ux=_full(nx, ny, 0.02 * c * gen.uniform(0.8, 1.2)), uy=_full(nx, ny, -0.01 * c * gen.uniform(0.8, 1.2)),
                    b=None)
        return dict(params=p, bcs=[], init=init, q3=None)
    # layered flow between walls, liquid below
    H = 0.5e-3
    dx = H / ny
    W = max(25e-6, 4 * dx)
    zl, zg = fl["rho_l"] * fl["nu_l"], fl["rho_g"] * fl["nu_g"]
    yy = (torch.arange(ny, dtype=torch.float64, device="cuda")[:, None] + 0.5) * dx
    phi = (0.5 - 0.5 * torch.tanh((2 * yy - H * float(gen.uniform(0.9, 1.1))) / W)).expand(ny, nx).contiguous()
    p.update(dx=dx, dt=dx / 100.0, W=W, nu_rule=1, Fb=(1e-4 * (zl + zg) / H ** 2, 0.0))
    bcs = [(s, lbm.LBM_BC_WALL, None, fl["rho_l"], lbm.LBM_TBC_NONE, None) for s in (2, 3)]
    s = yy / H
    init = dict(a=phi, ux=(4 * (s - s * s) * float(gen.uniform(0.8, 1.2))).expand(ny, nx).contiguous(),
                uy=(0.5 * torch.sin(math.pi * s) ** 2 * float(gen.uniform(0.8, 1.2))).expand(ny, nx).contiguous(), b=None)
    return dict(params=p, bcs=bcs, init=init, q3=None)


def _batch_specs(case):
    """Uneven channels as in the batched workload: nx ~ U{128..4096}, ny ~ U{32..512} (half
    as long in FP64), Pr 0.7 or 7, dt from a Mach rule clipped to relaxation times in
    [0.51, 2] dt."""
    gen = np.random.default_rng([case["spec"], 4])
    top = 4096 if case["prec"] == "f32" else 1024
    out = []
    for k in range(case["count"]):
        nx, ny = int(gen.integers(128, top + 1)), int(gen.integers(32, 513))
        Re, Pr = float(gen.uniform(10.0, 200.0)), float(gen.choice([0.7, 7.0]))
        nu, dx = Pr * ALPHA, 2.5e-6
        u_m = Re * nu / (2.0 * ny * dx)
        lo, hi = 0.01 * dx * dx / (3.0 * min(nu, ALPHA)), 0.5 * dx * dx / max(nu, ALPHA)
        dt = max(lo, min(0.1 * dx / (math.sqrt(3.0) * 1.5 * u_m), hi))
        out.append(dict(nx=nx, ny=ny, nu=nu, dx=dx, dt=dt, u_m=u_m))
    return out


def _batch_problems(case, seed):
    for k, sp in enumerate(_batch_specs(case)):
        yield _channel(dict(op="mrt", top="mrt"), np.random.default_rng([seed, 78, k]), **sp)


# ---------------------------------------------------------------------------
# A pass
# ---------------------------------------------------------------------------
_BITS = dict(rho=lbm.LBM_RHO, ux=lbm.LBM_UX, uy=lbm.LBM_UY, T=lbm.LBM_T, phi=lbm.LBM_PHI)


def _names(case):
    """The fields a case reads back, in the order of lbm_moments' planes."""
    if case["kind"] in ("bubble", "layered"):
        return ["rho", "ux", "uy", "phi"]
    if case["kind"] == "poiseuille":
        return ["rho", "ux", "uy"]
    return ["T"] if case["kind"] == "control" else ["ux", "uy", "T"]


def _mask(names):
    return sum(_BITS[k] for k in names)


def _precision(case):
    return lbm.LBM_FP64 if case["prec"] == "f64" else lbm.LBM_FP32DEV


def prepare(case, seed):
    names = _names(case)
    st = dict(case=case, names=names, mask=_mask(names))
    if case["kind"] == "batch":
        ws = list(_batch_problems(case, seed))
        st["stream"] = torch.cuda.Stream()
        st["batch"] = lbm.Batch([w["params"] for w in ws], precision=_precision(case), stream=st["stream"].cuda_stream)
        for ch, w in zip(st["batch"].channels, ws):
            for bc in w["bcs"]:
                ch.set_bc(*bc)
        st["inits"] = [w["init"] for w in ws]
        # all channels' velocities in one buffer and all temperatures in another
        nodes = [w["params"]["nx"] * w["params"]["ny"] for w in ws]
        st["out"] = [torch.empty(k * sum(nodes), dtype=torch.float64, device="cuda") for k in (2, 1)]
        st["views"] = [st["out"][0].split([2 * n for n in nodes]), st["out"][1].split(nodes)]
        return st
    w = _problem(case, seed)
    s = lbm.Solver(w["params"], precision=_precision(case))
    for bc in w["bcs"]:
        s.set_bc(*bc)
    if w["q3"] is not None:
        s.set_source(w["q3"], None)
    st.update(solver=s, init=w["init"], target=w.get("target"))
    if case["kind"] == "control":
        st["flux"] = [torch.from_numpy(bc[5]).pin_memory().numpy() for bc in w["bcs"][2:]]
        s.init(**w["init"])
    if case["kind"] != "adjoint":
        st["out"] = torch.empty((len(names), s.ny, s.nx), dtype=torch.float64, device="cuda")
    return st


def _handed_on(case, out):
    return out.to(torch.float32) if case["prec"] == "f32" else out


def _fields(st):
    out = lbm.lbm_moments(st["solver"].h, st["mask"], st["out"])
    return dict(zip(st["names"], _handed_on(st["case"], out)))


def run(st):
    case = st["case"]
    if case["kind"] == "batch":
        b = st["batch"]
        for ch, init in zip(b.channels, st["inits"]):
            ch.init(**init)
        b.step(case["steps"])
        for ch, u, T in zip(b.channels, *st["views"]):
            lbm.lbm_moments(ch.h, lbm.LBM_UX | lbm.LBM_UY, u)
            lbm.lbm_moments(ch.h, lbm.LBM_T, T)
        with torch.cuda.stream(st["stream"]):
            return dict(zip(("u", "T"), (_handed_on(case, v) for v in st["out"])))
    s = st["solver"]
    if case["kind"] == "adjoint":
        s.init(**st["init"])
        # dL/dnu is asked for in FP64 only: a sum of cancelling terms, of which the FP32 form
        # keeps three to five digits
        f64 = case["prec"] == "f64"
        loss, g3, gw, gn = lbm.lbm_adjoint(s.h, case["steps"], case["every"], st["target"], s.nx, s.ny, want_nu=f64)
        if f64:
            return dict(loss=np.float64(loss), g_q3=g3, g_qwall=gw, g_nu=np.float64(gn))
        return dict(loss=np.float32(loss), g_q3=g3.astype(np.float32), g_qwall=gw.astype(np.float32))
    if case["kind"] == "control":
        for side, q in zip((2, 3), st["flux"]):
            s.set_bc(side, lbm.LBM_BC_WALL, None, None, lbm.LBM_TBC_FLUX, q)
        s.step(1)
        return dict(integrals=s.integrals(), **_fields(st))
    s.init(**st["init"])
    s.step(case["steps"])
    return _fields(st)


# Floating-point operations of one node of one step (streaming none): momentum BGK or MRT,
# thermal D2Q5 / D2Q9, two-phase; the adjoint's reverse step is about twice the forward.
_FLOW, _TH5, _TH9, _MP = 140, 40, 110, 400


def work(case):
    kind, steps = case["kind"], case["steps"]
    if kind == "batch":
        nodes = sum(sp["nx"] * sp["ny"] for sp in _batch_specs(case))
    else:
        nodes = case["nx"] * case["ny"]
    out = 4 if case["prec"] == "f32" else 8
    R = 8 if case["prec"] == "f64" else 4
    if kind in ("bubble", "layered"):
        return dict(bytes=nodes * (3 * 8 + 4 * out), flops=float(_MP) * nodes * steps)
    if kind == "poiseuille":
        return dict(bytes=nodes * (2 * 8 + 3 * out), flops=float(_FLOW) * nodes * steps)
    if kind == "heated":
        return dict(bytes=nodes * (3 * 8 + 3 * out), flops=float(_FLOW + _TH9) * nodes * steps)
    if kind == "control":  # the state is the input and is returned updated
        return dict(bytes=nodes * (2 * 14 * R + out), flops=float(_FLOW + _TH5) * nodes * steps)
    if kind == "adjoint":  # fields and source in, source gradient out; forward and reverse
        return dict(bytes=nodes * (3 * 8 + R + out), flops=3.0 * (_FLOW + _TH5) * nodes * steps)
    return dict(bytes=nodes * (3 * 8 + 3 * out), flops=float(_FLOW + _TH5) * nodes * steps)


# ---------------------------------------------------------------------------
# The same in float64 with plain torch
# ---------------------------------------------------------------------------
C9 = [(0, 0), (1, 0), (0, 1), (-1, 0), (0, -1), (1, 1), (-1, 1), (-1, -1), (1, -1)]
W9 = [4 / 9] + [1 / 9] * 4 + [1 / 36] * 4
C5, W5 = C9[:5], [1 / 3] + [1 / 6] * 4


def _opp(C, q):
    return C.index((-C[q][0], -C[q][1]))


def _moment_rows(C):
    if len(C) == 5:
        return np.array([[1, x, y, 5 * (x * x + y * y) - 4, x * x - y * y] for x, y in C], dtype=float).T
    return np.array([[1, -4 + 3 * (x * x + y * y), 4 - 10.5 * (x * x + y * y) + 4.5 * (x * x + y * y) ** 2, x,
                      x * (3 * (x * x + y * y) - 5), y, y * (3 * (x * x + y * y) - 5), x * x - y * y, x * y] for x, y in C],
                    dtype=float).T


class _Lattice:
    def __init__(self, C, w):
        self.C, self.w, self.n = C, w, len(C)
        M = _moment_rows(C)
        self.M = torch.from_numpy(M).cuda()
        self.Mi = torch.from_numpy(np.linalg.inv(M)).cuda()

    def relax(self, f, feq, src, rates):
        """f - M^-1 S M (f - feq) + M^-1 (1 - S/2) M src; rates: one per moment (numbers or fields)."""
        sh = f.shape
        d = (self.M @ (f - feq).reshape(self.n, -1)).reshape(sh)
        m = [r * d[k] for k, r in enumerate(rates)]
        if src is not None:
            s = (self.M @ src.reshape(self.n, -1)).reshape(sh)
            m = [a - (1 - 0.5 * r) * s[k] for k, (a, r) in enumerate(zip(m, rates))]
        return f - (self.Mi @ torch.stack(m).reshape(self.n, -1)).reshape(sh)


def _bc_rules(bcs):
    sides = {s: dict(kind=0, tk=0, uw=None, rw=1.0, tw=None) for s in range(4)}
    for side, kind, uw, rw, tk, tw in bcs:
        dev = lambda v: None if v is None else (v if torch.is_tensor(v) else torch.from_numpy(np.asarray(v, float)).cuda())  # noqa: E731
        sides[side] = dict(kind=kind, tk=tk, uw=dev(uw), rw=rw, tw=dev(tw))
    return sides


def _edge(side):
    """Index of a side's nodes in a (ny, nx) field."""
    return [(slice(None), 0), (slice(None), -1), (0, slice(None)), (-1, slice(None))][side]


def _enters(side, c):
    return (c[0] > 0, c[0] < 0, c[1] > 0, c[1] < 0)[side]


def _wall_u(sd, n):
    if sd["uw"] is None:
        return 0.0, 0.0
    return sd["uw"][:n], sd["uw"][n:]


def _stream(L, fs, sides, key, c, cs2, rule):
    """Push fs one step; rule(side, q, o) gives the values of the links that enter through a
    side.  Symmetry sides first, then the x-sides, then the y-sides (which take corners)."""
    per = [sides[0][key] == 0 and sides[1][key] == 0, sides[2][key] == 0 and sides[3][key] == 0]
    sym = lbm.LBM_BC_SYMMETRY if key == "kind" else lbm.LBM_TBC_SYMMETRY
    out = []
    for q, (x, y) in enumerate(L.C):
        g = torch.roll(fs[q], (y, x), (0, 1))
        todo = [s for s in range(4) if _enters(s, (x, y)) and not per[s // 2]]
        for s in sorted(todo, key=lambda s: (sides[s][key] != sym, s)):
            if sides[s][key] == sym:
                v = torch.roll(fs[L.C.index((x, -y))], (x,), (1,))[_edge(s)]
            else:
                v = rule(s, q, _opp(L.C, q), g)
            g = g.clone()
            g[_edge(s)] = v
        out.append(g)
    return torch.stack(out)


class _Single:
    """Momentum (D2Q9) with an optional thermal lattice."""

    def __init__(self, w, nu=None, qd=None, sides=None):
        p = self.p = w["params"]
        self.c = p["dx"] / p["dt"]
        self.cs2 = self.c ** 2 / 3
        self.dt = p["dt"]
        self.F = _Lattice(C9, W9)
        self.G = None if not p["thermal"] else _Lattice(C5, W5) if p["thermal"] == 5 else self.F
        self.sides = sides or _bc_rules(w["bcs"])
        self.qd = qd
        tau = (p["nu"] if nu is None else nu) / self.cs2 + 0.5 * self.dt
        wn = 1 / tau
        sn = self.dt * wn
        sq = self.dt * (3 / self.dt) * (2 / self.dt - wn) / (3 / self.dt - wn)
        self.rates = [0.0, 1.0, 1.0, 0.0, sq, 0.0, sq, sn, sn] if p["flow_op"] == MRT else [sn] * 9
        if self.G:
            tT = p["k"] / (p["rho0"] * p["cp"]) / self.cs2 + 0.5 * self.dt
            sT = self.dt / tT
            mrt = [0.0, sT, sT, 1.0, 1.0] if p["thermal"] == 5 else [0.0, 1.0, 1.0, sT, 1.0, sT, 1.0, 1.0, 1.0]
            self.trates = mrt if p["thermal_op"] == MRT else [sT] * self.G.n
        i = w["init"]
        ny, nx = p["ny"], p["nx"]
        one = torch.ones((ny, nx), dtype=torch.float64, device="cuda")
        rho = one * p["rho0"] if i["a"] is None else i["a"]
        ux, uy = (torch.zeros_like(one) if i[k] is None else i[k] for k in ("ux", "uy"))
        self.f = self.feq(rho, ux, uy)
        if self.G:
            self.g = self.geq(one * p["T0"] if i["b"] is None else i["b"], ux, uy)

    def feq(self, rho, ux, uy):
        out, usq = [], (ux * ux + uy * uy) / (2 * self.cs2)
        for (x, y), w in zip(C9, W9):
            cu = self.c * (x * ux + y * uy) / self.cs2
            out.append(w * rho * (1 + cu + 0.5 * cu * cu - usq))
        return torch.stack(out)

    def geq(self, T, ux, uy):
        return torch.stack([w * T * (1 + self.c * (x * ux + y * uy) / self.cs2) for (x, y), w in zip(self.G.C, self.G.w)])

    def moments(self):
        p, f = self.p, self.f
        rho = f.sum(0)
        T = None
        Fx, Fy = p.get("Fb", (0.0, 0.0))
        if self.G:
            T = self.g.sum(0) + (0.0 if self.qd is None else 0.5 * self.dt * self.qd)
            if p.get("beta_exp"):
                k = -p["rho_ref"] * p["beta_exp"] * (T - p["T_ref"])
                Fx, Fy = Fx + k * p["gravity"][0], Fy + k * p["gravity"][1]
        jx = self.c * (f[1] - f[3] + f[5] - f[6] - f[7] + f[8])
        jy = self.c * (f[2] - f[4] + f[5] + f[6] - f[7] - f[8])
        return rho, (jx + 0.5 * self.dt * Fx) / rho, (jy + 0.5 * self.dt * Fy) / rho, T, Fx, Fy

    def step(self):
        rho, ux, uy, T, Fx, Fy = self.moments()
        p, c, cs2 = self.p, self.c, self.cs2
        src = None
        if torch.is_tensor(Fx) or Fx or Fy:
            src = torch.stack([self.dt * w * (((c * x - ux) * Fx + (c * y - uy) * Fy) / cs2 + c * (x * ux + y * uy) * c * (x * Fx + y * Fy) / cs2 ** 2)
                               for (x, y), w in zip(C9, W9)])
        fs = self.F.relax(self.f, self.feq(rho, ux, uy), src, self.rates)

        def f_rule(s, q, o, g):
            sd = self.sides[s]
            x, y = C9[o][0] * c, C9[o][1] * c
            if sd["kind"] == lbm.LBM_BC_PRESSURE:  # side 1 (x+) in these cases
                a, b = _edge(1), (slice(None), -2)
                wx, wy = 1.5 * ux[a] - 0.5 * ux[b], 1.5 * uy[a] - 0.5 * uy[b]
                cu = x * wx + y * wy
                return -fs[o][a] + 2 * W9[o] * sd["rw"] * (1 + cu * cu / (2 * cs2 ** 2) - (wx * wx + wy * wy) / (2 * cs2))
            wx, wy = _wall_u(sd, p["ny"] if s < 2 else p["nx"])
            return fs[o][_edge(s)] - 2 * W9[o] * sd["rw"] * (x * wx + y * wy) / cs2

        self.f = _stream(self.F, fs, self.sides, "kind", c, cs2, f_rule)
        if not self.G:
            return
        G = self.G
        tsrc = None if self.qd is None else torch.stack([self.dt * w * self.qd for w in G.w])
        gs = G.relax(self.g, self.geq(T, ux, uy), tsrc, self.trates)
        flux = self.dt / (p["dx"] * p["rho0"] * p["cp"])

        def g_rule(s, q, o, g):
            sd = self.sides[s]
            if sd["tk"] == lbm.LBM_TBC_OUTFLOW:
                return g[:, -2]
            if sd["tk"] == lbm.LBM_TBC_TEMP:
                wx, wy = _wall_u(sd, p["ny"] if s < 2 else p["nx"])
                cu = c * (G.C[o][0] * wx + G.C[o][1] * wy)
                return -gs[o][_edge(s)] + 2 * G.w[o] * sd["tw"] * (1 + cu * cu / (2 * cs2 ** 2) - (wx * wx + wy * wy) / (2 * cs2))
            return gs[o][_edge(s)] + (6 * W9[o] if G.n == 9 else 1.0) * flux * sd["tw"]

        self.g = _stream(G, gs, self.sides, "tk", c, cs2, g_rule)


class _TwoPhase:
    def __init__(self, w):
        p = self.p = w["params"]
        self.Z, self.H = _Lattice(C9, W9), _Lattice(C5, W5)
        self.c = p["dx"] / p["dt"]
        self.cs2 = self.c ** 2 / 3
        self.wall = bool(w["bcs"])
        self.sides = _bc_rules(w["bcs"])
        i, phi = w["init"], w["init"]["a"]
        ux, uy, pr = (torch.zeros_like(phi) if i[k] is None else i[k] for k in ("ux", "uy", "b"))
        rho = p["rho_g"] + phi * (p["rho_l"] - p["rho_g"])
        self.z = self.zeq(rho, ux, uy, pr)
        self.h = self.heq(phi, ux, uy)
        self.prev = (phi * ux, phi * uy)

    def zeq(self, rho, ux, uy, pr):
        out, usq = [], (ux * ux + uy * uy) / (2 * self.cs2)
        for q, ((x, y), w) in enumerate(zip(C9, W9)):
            cu = self.c * (x * ux + y * uy) / self.cs2
            out.append(pr / self.cs2 * (w - (q == 0)) + rho * w * (cu + 0.5 * cu * cu - usq))
        return torch.stack(out)

    def heq(self, phi, ux, uy):
        return torch.stack([w * phi * (1 + self.c * (x * ux + y * uy) / self.cs2) for (x, y), w in zip(C5, W5)])

    def _at(self, a, x, y):
        """a at the neighbour (i + x, j + y): periodic, or mirrored at the walls."""
        if not self.wall or not y:
            return torch.roll(a, (-y, -x), (0, 1))
        b = torch.cat([a[:1], a[:-1]]) if y < 0 else torch.cat([a[1:], a[-1:]])
        return torch.roll(b, (-x,), (1,))

    def moments(self):
        p, z, cs2, dt = self.p, self.z, self.cs2, self.p["dt"]
        phi = self.h.sum(0)
        nb = [self._at(phi, x, y) for x, y in C9]
        gx = 3 / p["dx"] * sum(w * x * n for (x, y), w, n in zip(C9, W9, nb) if x)
        gy = 3 / p["dx"] * sum(w * y * n for (x, y), w, n in zip(C9, W9, nb) if y)
        lap = 6 / p["dx"] ** 2 * sum(w * (n - phi) for w, n in zip(W9[1:], nb[1:]))
        kappa, beta = 1.5 * p["sigma"] * p["W"], 12 * p["sigma"] / p["W"]
        mu = 4 * beta * phi * (phi - 1) * (phi - 0.5) - kappa * lap
        Fb = p.get("Fb", (0.0, 0.0))
        Fx, Fy = mu * gx + Fb[0], mu * gy + Fb[1]
        dr = p["rho_l"] - p["rho_g"]
        rho = p["rho_g"] + phi * dr
        ux = (self.c * (z[1] - z[3] + z[5] - z[6] - z[7] + z[8]) + 0.5 * dt * Fx) / rho
        uy = (self.c * (z[2] - z[4] + z[5] + z[6] - z[7] - z[8]) + 0.5 * dt * Fy) / rho
        s0 = -4 / 9 * (ux * ux + uy * uy) / (2 * cs2)
        pr = cs2 * 1.8 * (z[1:].sum(0) + 0.5 * dt * dr * (ux * gx + uy * gy) + rho * s0)
        return rho, ux, uy, pr, phi, gx, gy, Fx, Fy

    def step(self):
        p, c, cs2, dt = self.p, self.c, self.cs2, self.p["dt"]
        rho, ux, uy, pr, phi, gx, gy, Fx, Fy = self.moments()
        dr = p["rho_l"] - p["rho_g"]
        if p.get("nu_rule", 0):
            zl, zg = p["rho_l"] * p["nu_l"], p["rho_g"] * p["nu_g"]
            nu = (zg + phi * (zl - zg)) / rho
        else:
            nu = p["nu_g"] + phi * (p["nu_l"] - p["nu_g"])
        sn = 1 / (nu / (cs2 * dt) + 0.5)
        # interface: advection of phi u and the sharpening flux along the normal
        g2 = gx * gx + gy * gy
        rn = torch.where(g2 > 0, 1 / torch.sqrt(torch.where(g2 > 0, g2, torch.ones_like(g2))), torch.zeros_like(g2))
        pu = (phi * ux, phi * uy)
        a = 4 * cs2 / p["W"] * phi * (1 - phi)
        ax, ay = (pu[0] - self.prev[0]) / dt + a * gx * rn, (pu[1] - self.prev[1]) / dt + a * gy * rn
        self.prev = pu
        om = dt / (p["mobility"] / cs2 + 0.5 * dt)
        src = torch.stack([dt * w * c * (x * ax + y * ay) / cs2 for (x, y), w in zip(C5, W5)])
        hs = self.H.relax(self.h, self.heq(phi, ux, uy), src, [om] * 5)
        src = torch.stack([dt * w * (c * (x * Fx + y * Fy) + c * (x * ux + y * uy) * c * dr * (x * gx + y * gy)) / cs2
                           for (x, y), w in zip(C9, W9)])
        rates = [sn] * 9
        if p["z_op"] == MRT:
            sq = 3 * (2 - sn) / (3 - sn)
            rates = [1.0, 1.0, 1.0, 1.0, sq, 1.0, sq, sn, sn]
        zs = self.Z.relax(self.z, self.zeq(rho, ux, uy, pr), src, rates)
        self.h = _stream(self.H, hs, self.sides, "kind", c, cs2, lambda s, q, o, g: hs[o][_edge(s)])
        self.z = _stream(self.Z, zs, self.sides, "kind", c, cs2, lambda s, q, o, g: zs[o][_edge(s)])


def _exact_adjoint(case, w):
    p = w["params"]
    qd = (w["q3"] / (p["rho0"] * p["cp"])).requires_grad_()
    nu = torch.tensor(p["nu"], dtype=torch.float64, device="cuda", requires_grad=True)
    sides = _bc_rules(w["bcs"])
    for s in (2, 3):
        sides[s]["tw"].requires_grad_()

    sim = _Single(w, nu.detach(), qd.detach(), sides)

    def segment(f, g, q, n, t2, t3, k):
        sd = {0: sides[0], 1: sides[1], 2: dict(sides[2], tw=t2), 3: dict(sides[3], tw=t3)}
        m = _Single(w, n, q, sd)
        m.f, m.g = f, g
        for _ in range(k):
            m.step()
        return m.f, m.g

    from torch.utils.checkpoint import checkpoint
    f, g, left = sim.f, sim.g, case["steps"]
    while left:
        k = min(10, left)
        f, g = checkpoint(segment, f, g, qd, nu, sides[2]["tw"], sides[3]["tw"], k, use_reentrant=False)
        left -= k
    T = g.sum(0) + 0.5 * p["dt"] * qd
    loss = ((T[:, -1] - torch.from_numpy(w["target"]).cuda()) ** 2).mean()
    g3, t2, t3, gn = torch.autograd.grad(loss, [qd, sides[2]["tw"], sides[3]["tw"], nu])
    out = dict(loss=loss.detach(), g_q3=g3 / (p["rho0"] * p["cp"]), g_qwall=torch.stack([t2, t3]))
    return dict(out, g_nu=gn) if case["prec"] == "f64" else out


def exact(case, seed):
    if case["kind"] == "batch":
        u, temps = [], []
        for w in _batch_problems(case, seed):
            m = _Single(w)
            for _ in range(case["steps"]):
                m.step()
            _, ux, uy, T, _, _ = m.moments()
            u += [ux.reshape(-1), uy.reshape(-1)]
            temps.append(T.reshape(-1))
        return dict(u=torch.cat(u), T=torch.cat(temps))
    w = _problem(case, seed)
    if case["kind"] == "adjoint":
        return _exact_adjoint(case, w)
    two = case["kind"] in ("bubble", "layered")
    m = _TwoPhase(w) if two else _Single(w)
    for _ in range(case["steps"]):
        m.step()
    v = m.moments()
    fields = dict(zip(("rho", "ux", "uy"), v), **({"phi": v[4]} if two else {"T": v[3]}))
    out = {k: fields[k] for k in _names(case)}
    if case["kind"] == "control":
        dx = w["params"]["dx"]
        umax = torch.sqrt(v[1] ** 2 + v[2] ** 2).max()
        out["integrals"] = [float(v[0].sum()) * dx * dx, 0.0, float(umax), 0.0]
    return out
