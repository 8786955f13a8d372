"""The work that a user of this library has it do, as cases that can be timed and checked.

Each case goes through the public Python binding (``api``, ``autograd``, ``closure``), on
synthetic flows of the shapes and recipes of ``config.WORKLOADS``: isentropic vortices and
random-phase solenoidal turbulence.  ``exact`` restates the discretisation in plain torch
in 64 bits (its adjoint by automatic differentiation) and uses none of the library.

Kinds of case:
  sweep     forward run, checkpointed reverse run, energy and sigma_1 series
  steps     one primal step and one adjoint step, as a caller with its own time loop makes
  autograd  loss and gradients of a batch of boxes with a parametrised source
  diagnose  sigma_1 field, the rule's viscosity, adjoint energy of one state
  infer     learned closure: features and viscosity of every cell of one state
  train     learned closure: one Adam step on a minibatch of cells
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_1511_06959_gb300 import api, autograd, closure, config

GAMMA, PR, CFL = 1.4, 0.72, 0.5
ROE_DELTA = 0.1
SCHEDULES = {"all": api.NS_CKPT_ALL, "stride": api.NS_CKPT_STRIDE, "revolve": api.NS_CKPT_REVOLVE}
BCS = {"periodic": api.NS_BC_PERIODIC, "inout": api.NS_BC_INOUT, "walls": api.NS_BC_WALLS,
       "inout_walls": api.NS_BC_INOUT_WALLS}
WALL_E = 1.0 / (GAMMA * (GAMMA - 1.0))   # the free stream's internal energy

BASE = {"kind": "steps", "nx": 128, "ny": 64, "nz": 64, "batch": 1, "precision": "mixed", "scheme": "rk4",
        "flux": "central", "bc": "periodic", "flow": "turbulence", "mach": 0.9, "Re": 1e4, "rms": 0.1,
        "lam_tilde": 0.1, "nsteps": 0, "schedule": "all", "param": 0, "graph": False, "record": False,
        "source": False, "nphi": 0, "minibatch": 0}


def _case(name=None, **kw):
    c = {**BASE, **kw}
    if name is not None:
        c["name"] = name
    return c


def _workload(w, **kw):
    d = {"nx": w.nx, "ny": w.ny, "nz": w.nz, "batch": w.batch, "flow": w.kind, "mach": w.mach, "Re": w.Re,
         "rms": w.rms, "lam_tilde": w.lam_tilde, "schedule": w.schedule, "param": w.param}
    return {**d, **kw}


def listed():
    W = config.WORKLOADS
    return [
        # a 2D study: thousands of short launches, where latency counts; captured once, replayed
        _case("vortex64_sweep_graph", **_workload(W["vortex64"], kind="sweep", nsteps=100, graph=True)),
        # the same box in the verification precision, by a direct call
        _case("vortex64_sweep_fp64", **_workload(W["vortex64"], kind="sweep", nsteps=50, precision="fp64")),
        # production: a transonic box, stride checkpoints, stabilised, with its diagnostics
        _case("box128_sweep", **_workload(W["box128"], kind="sweep", nsteps=100, param=25, graph=True, record=True)),
        # the reference gradient of that box in FP64
        _case("box128_sweep_fp64", **_workload(W["box128"], kind="sweep", nsteps=10, param=5, precision="fp64",
                                               record=True)),
        # an optimiser's iteration: eight boxes, loss and gradients for 64 source parameters
        _case("column96_autograd", **_workload(W["column96"], kind="autograd", nsteps=20, nphi=64)),
        # a caller's own time loop on a box no tile divides, with a source and its sensitivity
        _case("ragged_steps", nx=131, ny=67, nz=41, source=True),
        # the largest box: one step each way, fields far beyond the L2 cache
        _case("box512_steps", **_workload(W["box512"])),
        # a duct: inflow, outflow and walls
        _case("channel_steps", nx=96, ny=48, nz=48, bc="inout_walls", mach=0.5, flow="vortex", Re=1e3),
        # the paper's own scheme: Roe flux and SSP-RK3
        _case("roe_ssprk3_steps", flux="roe", scheme="ssprk3"),
        # growth analysis of one state
        _case("box128_diagnose", kind="diagnose"),
        # the learned closure: a batch of boxes, and one training step
        _case("column96_infer", **_workload(W["column96"], kind="infer", lam_tilde=0.5)),
        _case("closure_train", kind="train", nx=64, ny=64, nz=1, flow="vortex", mach=0.5, Re=1e3, minibatch=4096),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["sweep", "sweep", "steps", "steps", "steps", "autograd", "diagnose", "infer", "train"])
    flat = rng.random() < 0.2
    c = _case(kind=kind, precision="mixed" if rng.random() < 0.65 else "fp64",
              scheme=rng.choice(["rk4", "rk4", "rk4", "ssprk3"]))
    if flat:
        c.update(nx=_log_int(rng, 24, 400), ny=_log_int(rng, 24, 400), nz=1, flow="vortex", mach=0.5, Re=1e3)
    else:
        c.update(nx=_log_int(rng, 24, 320), ny=_log_int(rng, 12, 160), nz=_log_int(rng, 6, 96))
        if rng.random() < 0.4:
            c.update(flow="vortex", mach=0.5, Re=1e3)
    cells = c["nx"] * c["ny"] * c["nz"]
    if rng.random() < 0.3:
        c["flux"] = "roe"
    c["lam_tilde"] = rng.choice([0.0, 0.1, 0.1])
    if kind == "train":
        return _case(kind="train", nx=64, ny=64, nz=1, flow="vortex", mach=0.5, Re=1e3,
                     minibatch=_log_int(rng, 256, 16384))
    if kind == "steps":
        c["source"] = rng.random() < 0.3
        if rng.random() < 0.25:
            c["bc"] = rng.choice(["inout", "walls", "inout_walls"])
        return c
    if kind in ("diagnose", "infer"):
        c.update(batch=rng.choice([1, 1, 2, 4]), lam_tilde=0.1, flux="central")
        if kind == "infer":
            c["precision"] = "mixed"
        return c
    # whole calls: cell-steps within those of the listed ones
    budget = (12e6 if c["precision"] == "mixed" else 3e6) / (4 if c["flux"] == "roe" else 1)
    c["nsteps"] = max(3, min(60, int(budget / cells)))
    if kind == "autograd":
        c.update(nphi=rng.choice([16, 64]), batch=rng.choice([1, 2, 4]), lam_tilde=0.0)
        c["nsteps"] = max(2, c["nsteps"] // (2 * c["batch"]))
        return c
    c["schedule"] = rng.choice(["all", "stride", "stride", "revolve"])
    c["param"] = {"all": 0, "stride": max(2, c["nsteps"] // 4), "revolve": max(1, c["nsteps"] // 5)}[c["schedule"]]
    c["graph"] = rng.random() < 0.5
    c["record"] = rng.random() < 0.5
    return c


# ------------------------------------------------------------------------------------
# inputs
# ------------------------------------------------------------------------------------
def _gen(seed, k):
    return torch.Generator(device="cuda").manual_seed(1000003 * int(seed) + k)


def _randn(gen, *shape):
    return torch.randn(*shape, generator=gen, device="cuda", dtype=torch.float64)


def _flow(case, seed):
    """w[batch, 5, nz, ny, nx] of the case's flow: sound speed 1, length 1 along x, cubic cells."""
    nx, ny, nz = case["nx"], case["ny"], case["nz"]
    d = 1.0 / nx
    shape = (nz, ny, nx)
    out = torch.empty((case["batch"], 5) + shape, dtype=torch.float64, device="cuda")
    for b in range(case["batch"]):
        g = _gen(seed, 10 + b)
        if case["flow"] == "vortex":
            ax = [(torch.arange(n, device="cuda", dtype=torch.float64) + 0.5) * d for n in (nz, ny, nx)]
            _, Y, X = torch.meshgrid(*ax, indexing="ij")
            L, R, beta = (1.0, ny * d), 0.1, 5.0
            dx = torch.remainder(X - 0.5 * L[0] + 0.5 * L[0], L[0]) - 0.5 * L[0]
            dy = torch.remainder(Y - 0.5 * L[1] + 0.5 * L[1], L[1]) - 0.5 * L[1]
            f = torch.exp(0.5 * (1.0 - (dx ** 2 + dy ** 2) / R ** 2))
            T = 1.0 - (GAMMA - 1.0) * beta ** 2 / (8.0 * GAMMA * math.pi ** 2) * f ** 2
            rho = T ** (1.0 / (GAMMA - 1.0))
            p = rho * T / GAMMA
            a = beta / (2.0 * math.pi * math.sqrt(GAMMA))
            u = torch.stack([case["mach"] - a * dy / R * f, a * dx / R * f, torch.zeros_like(f)])
            rho = rho * (1.0 + 1e-3 * _randn(g, *shape))
            noise = 1e-3 * case["mach"] * _randn(g, 3, *shape)
            if nz == 1:
                noise[2] = 0.0
            u = u + noise
        else:
            # Fourier shells 2..16 of k L_y / 2 pi, |u_k|^2 ~ k^(-11/3), projected divergence-free
            ks = [torch.fft.fftfreq(n, d=1.0 / n, device="cuda", dtype=torch.float64) * (2 * math.pi / (n * d))
                  for n in (nz, ny, nx)]
            K = torch.stack(torch.meshgrid(*ks, indexing="ij")[::-1])
            k2 = (K ** 2).sum(0)
            kn = k2.sqrt() * (ny * d) / (2 * math.pi)
            amp = torch.where((kn >= 2) & (kn <= 16), kn.clamp(min=1.0) ** (-11.0 / 6.0), torch.zeros_like(kn))
            for axis, n in enumerate(shape):
                if n % 2 == 0:
                    amp.select(axis, n // 2).zero_()
            uh = torch.complex(_randn(g, 3, *shape), _randn(g, 3, *shape)) * amp
            uh = uh - K * ((K * uh).sum(0) / k2.clamp(min=1e-300))
            u = torch.fft.ifftn(uh, dim=(1, 2, 3)).real
            u = u - u.mean(dim=(1, 2, 3), keepdim=True)
            u = u * (case["rms"] * case["mach"] / u.square().mean().sqrt().clamp(min=1e-300))
            u[0] += case["mach"]
            rho = torch.ones(shape, dtype=torch.float64, device="cuda")
            p = torch.full(shape, 1.0 / GAMMA, dtype=torch.float64, device="cuda")
        out[b, 0] = rho
        out[b, 1:4] = rho * u
        out[b, 4] = p / (GAMMA - 1.0) + 0.5 * rho * u.square().sum(0)
    return out


def _smooth(gen, *shape):
    """Noise smoothed over neighbouring cells, as adjoint and source fields look."""
    a = _randn(gen, *shape)
    for ax in (-1, -2, -3):
        a = 0.5 * a + 0.25 * (a.roll(1, ax) + a.roll(-1, ax))
    return a


def _bumps(case):
    """phi[nphi, nz, ny, nx]: Gaussian source shapes at x = L_x / 4 on a grid in (y, z), or along y in 2D."""
    nx, ny, nz, n = case["nx"], case["ny"], case["nz"], case["nphi"]
    d = 1.0 / nx
    Z, Y, X = torch.meshgrid(*[(torch.arange(m, device="cuda", dtype=torch.float64) + 0.5) * d
                               for m in (nz, ny, nx)], indexing="ij")
    s = int(round(math.sqrt(n)))
    mid = [((m + 0.5) / n, 0.5) for m in range(n)] if nz == 1 else [((i + 0.5) / s, (j + 0.5) / s)
                                                                    for j in range(s) for i in range(s)]

    def dist2(a, c, L):
        return (torch.remainder(a - c * L + 0.5 * L, L) - 0.5 * L) ** 2

    r = [dist2(X, 0.25, 1.0) + dist2(Y, cy, ny * d) + (dist2(Z, cz, nz * d) if nz > 1 else 0.0) for cy, cz in mid]
    return torch.stack([torch.exp(-0.5 * q / (3.0 * d) ** 2) for q in r])


def _dt(case, w):
    q = _primitives(w)
    speed = q[1].square().add(q[2].square()).add(q[3].square()).sqrt() + (GAMMA * q[5] / q[0]).sqrt()
    return CFL / case["nx"] / float(speed.max())


def _inputs(case, seed):
    """Every input tensor of the case, from the seed alone."""
    w = _flow(case, seed)
    dx = 1.0 / case["nx"]
    x = {"w": w, "dt": _dt(case, w)}
    g = _gen(seed, 1)
    if case["kind"] in ("steps", "diagnose"):
        x["lam"] = 1e-6 * _smooth(g, *w.shape)
    if case["kind"] == "steps" and case["lam_tilde"] > 0:
        nu = case["lam_tilde"] * dx ** 2 * _sigma1(w, _Constants(case, 0.0))
        x["nu"] = nu if case["precision"] == "fp64" else nu.float()
    if case["kind"] == "steps" and case["source"]:
        x["s"] = 0.02 * _smooth(g, *w.shape)
        x["sbar"] = 1e-6 * _smooth(g, *w.shape)
    if case["kind"] == "autograd":
        x["phi"] = _bumps(case)
        x["theta"] = 0.02 * _randn(g, x["phi"].shape[0])
    if case["kind"] in ("infer", "train"):
        x["params"] = closure.init_params(int(seed), 0.3)
    if case["kind"] == "train":
        n = 16 * 4096
        x["feat"] = torch.zeros((n, 16), dtype=torch.float32, device="cuda")
        x["feat"][:, :14] = torch.randn(n, 14, generator=g, device="cuda")
        x["target"] = torch.randn(n, generator=g, device="cuda").abs()
        x["idx"] = torch.randint(0, n, (case["minibatch"],), generator=g, device="cuda", dtype=torch.int32)
    return x


# ------------------------------------------------------------------------------------
# the library
# ------------------------------------------------------------------------------------
def prepare(case, seed):
    x = _inputs(case, seed)
    w, dx = x["w"], 1.0 / case["nx"]
    c = _Constants(case, x["dt"])
    S = api.Solver(case["nx"], case["ny"], case["nz"], dx, gamma=GAMMA, mu=c.mu, Pr=PR, dt=x["dt"],
                   precision=api.NS_FP64 if case["precision"] == "fp64" else api.NS_MIXED, plane_i=c.plane,
                   pt_in=c.pt_in, batch=case["batch"],
                   scheme=api.NS_SSPRK3 if case["scheme"] == "ssprk3" else api.NS_RK4,
                   flux=api.NS_FLUX_ROE if case["flux"] == "roe" else api.NS_FLUX_CENTRAL, roe_delta=ROE_DELTA)
    if case["bc"] != "periodic":
        S.set_boundaries(BCS[case["bc"]], far=c.far, wall_e=(WALL_E, WALL_E))
    st = {"case": case, "S": S, **x}
    cells, B = S.cells * S.batch, S.batch
    f32, f64 = ({"dtype": t, "device": "cuda"} for t in (torch.float32, torch.float64))
    kind = case["kind"]
    if kind == "sweep":
        N = case["nsteps"]
        st["opts"] = S.run_opts(N, SCHEDULES[case["schedule"]], case["param"], case["lam_tilde"] * dx ** 2, 0.0,
                                case["record"], case["record"])
        st["arena"] = torch.empty(S.arena_bytes(st["opts"]), dtype=torch.uint8, device="cuda")
        st["out"] = {"Jbar": torch.empty(B, **f64), "lam0": torch.empty_like(w), "sbar": torch.empty_like(w)}
        if case["record"]:
            st["out"].update(energy=torch.zeros((N + 1, B), **f64), sigma_stats=torch.zeros((N, B, 2), **f64))
        if case["graph"]:
            o = dict(st["out"])
            st["graph"] = S.adjoint_run_capture(w, st["opts"], st["arena"], o.pop("Jbar"), o.pop("lam0"), **o)
    elif kind == "steps":
        st["out"] = {"w1": torch.empty_like(w), "lam0": torch.empty_like(w)}
        if "s" in x:
            st["out"]["sbar"] = x["sbar"]   # accumulated into, step by step
    elif kind == "autograd":
        st["w"] = w.requires_grad_(True)
        st["theta"] = x["theta"].requires_grad_(True)
        st["problem"] = autograd.SourceProblem(S, x["phi"], case["nsteps"])
    elif kind == "diagnose":
        t = f64 if case["precision"] == "fp64" else f32
        st["out"] = {"sigma1": torch.empty(cells, **t), "nu": torch.empty(cells, **t),
                     "stats": torch.empty((B, 2), **f64), "energy": torch.empty(B, **f64)}
    elif kind == "infer":
        st["net"] = closure.Network(S, x["params"])
        st["out"] = {"feat": torch.empty((cells, 16), **f32), "sigma1": torch.empty(cells, **f32),
                     "nu": torch.empty(cells, **f32)}
    else:
        st["net"] = closure.Network(S, x["params"])
        n = api.NS_MLP_PARAMS
        st["out"] = {"loss": torch.empty(1, **f32), "params": torch.empty(n, **f32), "m": torch.empty(n, **f32),
                     "v": torch.empty(n, **f32)}
    return st


def run(st):
    case, S, kind, o = st["case"], st["S"], st["case"]["kind"], st.get("out")
    dx = 1.0 / case["nx"]
    if kind == "sweep":
        if "graph" in st:
            st["graph"].launch()
        else:
            S.adjoint_run(st["w"], st["opts"], st["arena"], o["Jbar"], o["lam0"], sbar=o["sbar"],
                          energy=o.get("energy"), sigma_stats=o.get("sigma_stats"))
        return o
    if kind == "steps":
        S.primal_step(st["w"], o["w1"], st.get("s"))
        S.adjoint_step(st["w"], st["lam"], o["lam0"], s=st.get("s"), nu=st.get("nu"), sbar=o.get("sbar"))
        return o
    if kind == "autograd":
        J = st["problem"](st["w"], st["theta"])
        gw, gt = torch.autograd.grad(J.sum(), [st["w"], st["theta"]])
        return {"J": J.detach(), "gw": gw, "gtheta": gt}
    if kind == "diagnose":
        S.growth_sigma1(st["w"], o["sigma1"], o["stats"])
        S.add_adjoint_viscosity(o["sigma1"], case["lam_tilde"] * dx ** 2, o["nu"])
        S.adjoint_energy(st["w"], st["lam"], o["energy"])
        return o
    if kind == "infer":
        S.mlp_features(st["w"], o["feat"])
        S.growth_sigma1(st["w"], o["sigma1"])
        S.mlp_infer(st["net"].blob, o["feat"], o["sigma1"], case["lam_tilde"], o["nu"])
        return o
    net = st["net"]
    net.step += 1
    S.mlp_train_step(net.blob, st["feat"], st["target"], st["idx"], net.step, 2e-3, o["loss"])
    S.mlp_get_params(net.blob, o["params"])
    S.mlp_get_moment(net.blob, 1, o["m"])
    S.mlp_get_moment(net.blob, 2, o["v"])
    return o


def work(case):
    """Each input read once and each output written once; the arithmetic of the stages, per cell."""
    cells = case["nx"] * case["ny"] * case["nz"] * case["batch"]
    stages = 3 if case["scheme"] == "ssprk3" else 4
    rhs, adj = (500, 750) if case["flux"] == "central" else (1100, 2000)
    real = 8 if case["precision"] == "fp64" else 4
    nu = real if case["lam_tilde"] > 0 else 0
    kind = case["kind"]
    if kind == "sweep":
        return {"bytes": cells * 120, "flops": case["nsteps"] * cells * (stages * (rhs + adj) + (900 if nu else 0))}
    if kind == "steps":
        return {"bytes": cells * (160 + nu + (120 if case["source"] else 0)),
                "flops": cells * ((2 * stages - 1) * rhs + stages * adj)}
    if kind == "autograd":
        return {"bytes": cells * 80 + 8 * case["nphi"] * cells // case["batch"],
                "flops": case["nsteps"] * cells * stages * (rhs + adj)}
    if kind == "diagnose":
        return {"bytes": cells * (80 + 2 * real), "flops": cells * 1000}
    if kind == "infer":
        return {"bytes": cells * (40 + 64 + 4 + 4), "flops": cells * (2 * (16 * 64 + 64 * 64 + 64) + 1000)}
    n = case["minibatch"]
    return {"bytes": n * 72 + 6 * 4 * api.NS_MLP_PARAMS, "flops": n * 6 * (14 * 64 + 64 * 64 + 64)}


# ------------------------------------------------------------------------------------
# the same in plain torch, 64 bits
# ------------------------------------------------------------------------------------
class _Constants:
    def __init__(self, case, dt):
        self.dx, self.dt = 1.0 / case["nx"], dt
        self.mu = case["mach"] / case["Re"]
        self.alpha = GAMMA * self.mu / PR
        self.plane = (3 * case["nx"]) // 4
        self.pt_in = (1 / GAMMA) * (1 + 0.5 * (GAMMA - 1) * case["mach"] ** 2) ** (GAMMA / (GAMMA - 1))
        self.roe = case["flux"] == "roe"
        self.far = (1.0, case["mach"], 0.0, 0.0, 1.0 / GAMMA)
        self.inout = case["bc"] in ("inout", "inout_walls")
        self.walls = case["bc"] in ("walls", "inout_walls")
        self.flat = case["nz"] == 1
        if case["scheme"] == "ssprk3":
            self.A, self.b = [[], [1.0], [0.25, 0.25]], [1 / 6, 1 / 6, 2 / 3]
        else:
            self.A, self.b = [[], [0.5], [0.0, 0.5], [0.0, 0.0, 1.0]], [1 / 6, 1 / 3, 1 / 3, 1 / 6]


def _primitives(w):
    """rho, u1, u2, u3, e, p of w[batch, 5, ...]"""
    rho = w[:, 0]
    u = [w[:, 1 + k] / rho for k in range(3)]
    e = w[:, 4] / rho - 0.5 * (u[0] ** 2 + u[1] ** 2 + u[2] ** 2)
    return [rho, *u, e, (GAMMA - 1.0) * rho * e]


def _up(a, d):
    return a.roll(-1, -1 - d)


def _dn(a, d):
    return a.roll(1, -1 - d)


def _roe(q, d):
    """Roe dissipation of the face above each cell along d, with Harten's entropy fix."""
    L, R = q, [_up(a, d) for a in q]
    s = [x[0].sqrt() for x in (L, R)]
    wl, wr = s[0] / (s[0] + s[1]), s[1] / (s[0] + s[1])
    H = [GAMMA * x[4] + 0.5 * (x[1] ** 2 + x[2] ** 2 + x[3] ** 2) for x in (L, R)]
    u = [wl * L[1 + k] + wr * R[1 + k] for k in range(3)]
    Ht, rt = wl * H[0] + wr * H[1], s[0] * s[1]
    q2 = u[0] ** 2 + u[1] ** 2 + u[2] ** 2
    c = ((GAMMA - 1.0) * (Ht - 0.5 * q2)).sqrt()
    du = [R[1 + k] - L[1 + k] for k in range(3)]
    dp, delta = R[5] - L[5], ROE_DELTA * c
    a1 = (dp - rt * c * du[d]) / (2 * c * c)
    a3 = (dp + rt * c * du[d]) / (2 * c * c)
    a2 = R[0] - L[0] - dp / (c * c)
    l1, l2, l3 = (torch.where(v.abs() < delta, (v * v + delta * delta) / (2 * delta), v.abs())
                  for v in (u[d] - c, u[d], u[d] + c))
    D = [l1 * a1 + l2 * a2 + l3 * a3]
    for k in range(3):
        n = 1.0 if k == d else 0.0
        D.append(l1 * a1 * (u[k] - c * n) + l2 * a2 * u[k] + l3 * a3 * (u[k] + c * n) + l2 * rt * (du[k] - du[d] * n))
    D.append(l1 * a1 * (Ht - u[d] * c) + l2 * a2 * 0.5 * q2 + l3 * a3 * (Ht + u[d] * c)
             + l2 * rt * (u[0] * du[0] + u[1] * du[1] + u[2] * du[2] - u[d] * du[d]))
    return [0.5 * v for v in D]


def _with_ghosts(w, c):
    """w with one ghost layer on its bounded sides (columns first, then rows over them)."""
    g = GAMMA
    if c.inout:
        rf, uf, pf, k = c.far[0], c.far[1], c.far[4], 2.0 / (g - 1.0)
        cf = math.sqrt(g * pf / rf)
        cols = []
        for side, x in ((0, w[..., :1]), (1, w[..., -1:])):
            q = _primitives(x)
            cs = (g * q[5] / q[0]).sqrt()
            if side:
                Rp, Rm, ent, t = q[1] + k * cs, torch.full_like(cs, uf - k * cf), q[5] / q[0] ** g, (q[2], q[3])
            else:
                Rp, Rm, ent = torch.full_like(cs, uf + k * cf), q[1] - k * cs, torch.full_like(cs, pf / rf ** g)
                t = (torch.full_like(cs, c.far[2]), torch.full_like(cs, c.far[3]))
            ub, cb = 0.5 * (Rp + Rm), 0.25 * (g - 1.0) * (Rp - Rm)
            rho = (cb * cb / (g * ent)) ** (1.0 / (g - 1.0))
            E = rho * cb * cb / (g * (g - 1.0)) + 0.5 * rho * (ub ** 2 + t[0] ** 2 + t[1] ** 2)
            cols.append(torch.stack([rho, rho * ub, rho * t[0], rho * t[1], E], 1))
        w = torch.cat([cols[0], w, cols[1]], -1)
    if c.walls:
        rows = []
        for x in (w[..., :1, :], w[..., -1:, :]):
            q = _primitives(x)
            k2 = 0.5 * (q[1] ** 2 + q[2] ** 2 + q[3] ** 2)
            rows.append(torch.stack([q[0], -x[:, 1], -x[:, 2], -x[:, 3], q[0] * (2 * WALL_E - q[4] + k2)], 1))
        w = torch.cat([rows[0], w, rows[1]], -2)
    return w


def _crop(a, c):
    if c.inout:
        a = a[..., 1:-1]
    return a[..., 1:-1, :] if c.walls else a


def _residual(w, c):
    q = _primitives(_with_ghosts(w, c))
    rho, u, e, p = q[0], q[1:4], q[4], q[5]
    E = rho * (e + 0.5 * (u[0] ** 2 + u[1] ** 2 + u[2] ** 2))
    central = [[(_up(u[k], d) - _dn(u[k], d)) / (2 * c.dx) for d in range(3)] for k in range(3)]
    R = [0.0] * 5
    for d in range(3):
        m = rho * u[d]
        F = [m, *(m * u[k] + (p if k == d else 0.0) for k in range(3)), (E + p) * u[d]]
        g = [[(_up(u[k], d) - u[k]) / c.dx if l == d else 0.5 * (central[k][l] + _up(central[k][l], d))
              for l in range(3)] for k in range(3)]
        sig = [c.mu * (g[j][d] + g[d][j]) for j in range(3)]
        sig[d] = sig[d] - (2.0 / 3.0) * c.mu * (g[0][0] + g[1][1] + g[2][2])
        heat = c.alpha * (_up(e, d) - e) / c.dx
        Fv = [0.0, *sig, heat + sum(0.5 * (u[k] + _up(u[k], d)) * sig[k] for k in range(3))]
        D = _roe(q, d) if c.roe else [0.0] * 5
        for v in range(5):
            phi = 0.5 * (F[v] + _up(F[v], d)) - Fv[v] - D[v]
            R[v] = R[v] - (phi - _dn(phi, d)) / c.dx
    return _crop(torch.stack(R, 1), c)


def _stages(w, c, s):
    """stage states and stage slopes of one step"""
    W, k = [], []
    for row in c.A:
        x = w
        for a, kj in zip(row, k):
            x = x + c.dt * a * kj
        W.append(x)
        r = _residual(x, c)
        k.append(r if s is None else r + s)
    return W, k


def _step(w, c, s=None):
    _, k = _stages(w, c, s)
    return w + c.dt * sum(b * kj for b, kj in zip(c.b, k))


def _vjp(f, w, a):
    x = w.detach().requires_grad_(True)
    with torch.enable_grad():
        return torch.autograd.grad(f(x), x, a)[0]


def _viscosity(nu, a, c):
    """div(nu grad a) per component; no flux through the bounded sides' faces"""
    n, out = nu[:, None], 0.0
    for d in range(3):
        f = 0.5 * (n + _up(n, d)) * (_up(a, d) - a) / c.dx ** 2
        if (d == 0 and c.inout) or (d == 1 and c.walls):
            f = f.clone()
            f.select(-1 - d, -1).zero_()
        out = out + f - _dn(f, d)
    return out


def _adjoint_step(w, lam, c, s=None, nu=None):
    """lam^n and the sum of the stage seeds"""
    W, _ = _stages(w, c, s)
    n = len(W)
    g, seeds = [None] * n, 0.0
    for i in reversed(range(n)):
        a = c.b[i] * lam
        for m in range(i + 1, n):
            a = a + c.A[m][i] * g[m]
        a = c.dt * a
        g[i] = _vjp(lambda x: _residual(x, c), W[i], a)
        if nu is not None:
            g[i] = g[i] + _viscosity(nu, a, c)
        seeds = seeds + a
    return lam + sum(g), seeds


def _objective(w, c):
    nx = w.shape[-1]
    f = 0.5 * (w[..., (c.plane - 1) % nx] + w[..., c.plane % nx])
    q = _primitives(f)
    uu = q[1] ** 2 + q[2] ** 2 + q[3] ** 2
    pt = q[5] * (1 + 0.5 * (GAMMA - 1) * q[0] * uu / (GAMMA * q[5])) ** (GAMMA / (GAMMA - 1))
    return (q[0] * (c.pt_in - pt)).sum((1, 2)) / (q[0].sum((1, 2)) * c.pt_in)


def _sigma1(w, c):
    """Largest singular value of the growth matrix, by repeated squaring of M^T M."""
    q = _primitives(w)
    rho, u, p = q[0], q[1:4], q[5]
    cs = (GAMMA * p / rho).sqrt()
    a, b = math.sqrt((GAMMA - 1) / GAMMA) * cs, cs / math.sqrt(GAMMA)

    def grad(f):
        return [(_up(f, d) - _dn(f, d)) / (2 * c.dx) for d in range(3)]

    dr, dp, da, db, du = grad(rho), grad(p), grad(a), grad(b), [grad(v) for v in u]
    div = du[0][0] + du[1][1] + du[2][2]
    M = torch.zeros(w.shape[:1] + w.shape[2:] + (5, 5), dtype=w.dtype, device=w.device)
    for i in range(5):
        M[..., i, i] = 0.5 * div
    for j in range(3):
        M[..., 0, 1 + j] = 0.5 * db[j] - b / rho * dr[j]
        M[..., 1 + j, 0] = 0.5 * db[j]
        M[..., 1 + j, 4] = 0.5 * da[j] - a / (2 * p) * dp[j]
        M[..., 4, 1 + j] = 0.5 * da[j] - 2 / (GAMMA - 1) * da[j]
        for k in range(3):
            M[..., 1 + k, 1 + j] -= du[k][j]
    M[..., 0, 4] -= math.sqrt(GAMMA - 1) / 2 * div
    M[..., 4, 4] -= (GAMMA - 1) / 2 * div
    if c.flat:
        keep = [0, 1, 2, 4]
        M = M[..., keep, :][..., :, keep]
    B = M.transpose(-1, -2) @ M

    def trace(x):
        return x.diagonal(dim1=-2, dim2=-1).sum(-1)

    P = B
    for _ in range(30):
        P = P / trace(P).clamp(min=1e-300)[..., None, None]
        P = P @ P
    return (trace(B @ P) / trace(P).clamp(min=1e-300)).clamp(min=0).sqrt()


def _energy(w, lam, c):
    q = _primitives(w)
    rho, u, p = q[0], q[1:4], q[5]
    cs = (GAMMA * p / rho).sqrt()
    uu = u[0] ** 2 + u[1] ** 2 + u[2] ** 2
    y0 = lam[:, 0] + u[0] * lam[:, 1] + u[1] * lam[:, 2] + u[2] * lam[:, 3] + 0.5 * uu * lam[:, 4]
    y4 = lam[:, 4] / (GAMMA - 1)
    v0 = math.sqrt(GAMMA) * rho / cs * y0 + rho * cs / math.sqrt(GAMMA) * y4
    v4 = rho * cs * math.sqrt((GAMMA - 1) / GAMMA) * y4
    v = v0 ** 2 + v4 ** 2 + sum((rho * (lam[:, 1 + k] + u[k] * lam[:, 4])) ** 2 for k in range(3))
    return v.sum((1, 2, 3)) * c.dx ** 3


def _sweep(w0, c, N, s=None, nu_of=None, record=False):
    """Jbar, dJbar/dw0, dJbar/ds, and with record the energy and sigma_1 series"""
    W = [w0]
    for _ in range(N):
        W.append(_step(W[-1], c, s))
    one = torch.ones(w0.shape[0], dtype=w0.dtype, device=w0.device) / N
    J = sum(_objective(x, c) for x in W[1:]) / N
    lam = _vjp(lambda x: _objective(x, c), W[N], one)
    sbar = torch.zeros_like(w0)
    E, stats = [_energy(W[N], lam, c)], []
    for n in reversed(range(N)):
        sig = _sigma1(W[n], c) if nu_of is not None or record else None
        lam, seeds = _adjoint_step(W[n], lam, c, s, None if nu_of is None else nu_of(sig))
        if n >= 1:
            lam = lam + _vjp(lambda x: _objective(x, c), W[n], one)
        sbar = sbar + seeds
        if record:
            E.append(_energy(W[n], lam, c))
            stats.append(torch.stack([sig.amax((1, 2, 3)), sig.mean((1, 2, 3))], -1))
    out = {"Jbar": J, "lam0": lam, "sbar": sbar}
    if record:
        out.update(energy=torch.stack(E[::-1]), sigma_stats=torch.stack(stats[::-1]))
    return out


def _features(w, c):
    q = _primitives(w)
    m = [x.mean((1, 2, 3), keepdim=True) for x in q]
    cb = (GAMMA * m[5] / m[0]).sqrt()
    f = [(q[0] - m[0]) / (math.sqrt(GAMMA) * m[0])]
    f += [(q[1 + k] - m[1 + k]) / cb for k in range(3)]
    f += [(-cb / (m[0] * math.sqrt(GAMMA * (GAMMA - 1))) * (q[0] - m[0])
           + math.sqrt(GAMMA / (GAMMA - 1)) / (m[0] * cb) * (q[5] - m[5])) / cb]
    f += [(_up(q[1 + k], j) - _dn(q[1 + k], j)) / (2 * c.dx) / cb for k in range(3) for j in range(3)]
    f = torch.stack(f, -1).reshape(-1, 14)
    return torch.cat([f, torch.zeros_like(f[:, :2])], 1)


def _network(par, x):
    """softplus of the network on features x, its weights in the precision it keeps them in (BF16)"""
    def gelu(z):
        return 0.5 * z * (1 + torch.special.erf(z / math.sqrt(2)))
    b = {k: v.bfloat16().double() if k in ("W1", "W2", "w3") else v for k, v in par.items()}
    # rounded weights with the gradient of the master copies
    b = {k: par[k] + (b[k] - par[k]).detach() for k in par}
    h = gelu(gelu(x @ b["W1"] + b["b1"]) @ b["W2"] + b["b2"])
    return torch.nn.functional.softplus(h @ b["w3"] + b["b3"])


def exact(case, seed):
    x = _inputs(case, seed)
    c = _Constants(case, x["dt"])
    w, dx2, kind = x["w"], c.dx ** 2, case["kind"]
    shape = w.shape[:1] + w.shape[2:]
    if kind == "sweep":
        nu_of = (lambda sig: case["lam_tilde"] * dx2 * sig) if case["lam_tilde"] > 0 else None
        return _sweep(w, c, case["nsteps"], None, nu_of, case["record"])
    if kind == "steps":
        nu = x["nu"].double().reshape(shape) if "nu" in x else None
        lam, seeds = _adjoint_step(w, x["lam"], c, x.get("s"), nu)
        out = {"w1": _step(w, c, x.get("s")), "lam0": lam}
        if "s" in x:
            out["sbar"] = x["sbar"] + seeds
        return out
    if kind == "autograd":
        s = torch.zeros_like(w)
        s[:, 1] = torch.tensordot(x["theta"], x["phi"], dims=1)
        r = _sweep(w, c, case["nsteps"], s)
        g = torch.tensordot(x["phi"], r["sbar"][:, 1].sum(0), dims=3)
        return {"J": r["Jbar"], "gw": r["lam0"], "gtheta": g}
    if kind == "diagnose":
        sig = _sigma1(w, c)
        return {"sigma1": sig.reshape(-1), "nu": case["lam_tilde"] * dx2 * sig.reshape(-1),
                "stats": torch.stack([sig.amax((1, 2, 3)), sig.mean((1, 2, 3))], -1),
                "energy": _energy(w, x["lam"], c)}
    par = {k: torch.as_tensor(np.asarray(v, dtype=np.float32), device="cuda").double() for k, v in x["params"].items()}
    if kind == "infer":
        f, sig = _features(w, c), _sigma1(w, c).reshape(-1)
        nu = case["lam_tilde"] * dx2 * sig * _network(par, f[:, :14].bfloat16().double())
        return {"feat": f, "sigma1": sig, "nu": nu}
    i = x["idx"].long()
    leaf = {k: v.clone().requires_grad_(True) for k, v in par.items()}
    y = _network(leaf, x["feat"][i, :14].bfloat16().double())
    loss = (y - x["target"][i].double()).square().mean()
    g = torch.cat([t.reshape(-1) for t in torch.autograd.grad(loss, list(leaf.values()))])
    p = torch.cat([v.reshape(-1) for v in par.values()]) - 2e-3 * g / (g.abs() + 1e-8)
    return {"loss": loss.detach().reshape(1), "params": p, "m": 0.1 * g, "v": 0.001 * g * g}
