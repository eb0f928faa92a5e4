"""Timed cases: what a user of this library has it do, over the real range.

A case is a dict of plain values; ``prepare`` builds what a program has in
hand before the call (a cavity, an ensemble, a saved state, a wall field),
``run`` is one pass through the public entry points, and ``exact`` is the same
pass in 64-bit torch, written from the method's equations (D3Q19 and D3Q7
multiple-relaxation-time collision, pull streaming between two copies of the
state, the front's energy balance, the phase flip).

Kinds of a case:
  melt      advance a cavity by `steps` steps and read its fields; with
            `restore` the pass starts from a saved state and saves the state
            it ends in (small cavities, whose front would otherwise leave its
            place within the timing), without it the run goes on (large
            cavities: the front moves less than a node in ten thousand steps)
  ensemble  advance a batch of uneven cavities, from a saved state
  gradient  a loss of the final front and its gradient with respect to the
            heated-wall field and Ra (the torch.autograd form)
  loop      every step takes a new heated-wall field from page-locked host
            memory and sends the front and the liquid fraction back
  readout   fields, totals and Nusselt numbers of a state
"""
import ctypes
import math
import random

import numpy as np
import torch

from paper_1604_03478_gb300 import Cavity, Ensemble, _abi, autotune, inputs
from paper_1604_03478_gb300.autograd import melt_front

E19 = [(0, 0, 0), (1, 0, 0), (-1, 0, 0), (0, 1, 0), (0, -1, 0), (0, 0, 1), (0, 0, -1),
       (1, 1, 0), (-1, 1, 0), (1, -1, 0), (-1, -1, 0), (1, 0, 1), (-1, 0, 1), (1, 0, -1), (-1, 0, -1),
       (0, 1, 1), (0, -1, 1), (0, 1, -1), (0, -1, -1)]
E7 = E19[:7]
W19 = [1 / 3] + [1 / 18] * 6 + [1 / 36] * 12
W7 = [1 / 4] + [1 / 8] * 6
OPP19 = [E19.index((-x, -y, -z)) for x, y, z in E19]
OPP7 = OPP19[:7]
SIDE, BOTTOM = 0, 1  # heated wall y = 0 or z = 0
FP32, FP16 = 0, 1


def listed():
    convection = dict(Ra=1e6, Pr=0.02, Ste=0.05, Ma=0.1)
    return [
        # the smallest: conduction melting in a 32^3 cube, gravity off, where launches and latency count
        dict(name="conduction_32", kind="melt", nx=32, ny=32, nz=32, face=SIDE, precision=FP32, Ra=0.0, Pr=1.0,
             Ste=0.1, Ma=0.1, Tc=0.0, height=0.4, steps=50, restore=True),
        # convection melting at 128^3 early in the melt: a thin liquid layer, few nodes a column
        dict(name="convection_128_thin", kind="melt", nx=128, ny=128, nz=128, face=SIDE, precision=FP32, Ra=1e5,
             Pr=0.02, Ste=0.1, Ma=0.1, Tc=0.0, height=0.1, steps=64, restore=True),
        # a paper case (Table 1, case 1) at 96^3 in the middle of its melt
        dict(name="table1_96_mid", kind="melt", nx=96, ny=96, nz=96, face=SIDE, precision=FP32, Ra=25000.0,
             Pr=0.02, Ste=0.1, Ma=0.1, Tc=0.0, height=0.45, steps=64, restore=True),
        # a cavity of odd edges, heated at the bottom, late in the melt
        dict(name="ragged_101x75x83", kind="melt", nx=101, ny=75, nz=83, face=BOTTOM, precision=FP32, Ra=1e5,
             Pr=0.1, Ste=0.1, Ma=0.1, Tc=0.0, height=0.6, steps=40, restore=True),
        # the precision study: 256^3, side-heated with FP32 storage ...
        dict(name="side_256_fp32", kind="melt", nx=256, ny=256, nz=256, face=SIDE, precision=FP32, Tc=0.0,
             height=0.4, steps=20, restore=False, **convection),
        # ... and bottom-heated with shifted FP16 storage
        dict(name="bottom_256_fp16", kind="melt", nx=256, ny=256, nz=256, face=BOTTOM, precision=FP16, Tc=0.0,
             height=0.4, steps=8, restore=False, **convection),
        # heat conduction in a subcooled solid: every node of the cavity works
        dict(name="subcooled_256", kind="melt", nx=256, ny=256, nz=256, face=SIDE, precision=FP32, Tc=-0.25,
             height=0.4, steps=20, restore=False, **convection),
        # a step loop that talks to its host every step (a controller on the heated wall)
        dict(name="loop_256", kind="loop", nx=256, ny=256, nz=256, face=SIDE, precision=FP32, Tc=0.0, height=0.4,
             steps=20, **convection),
        # a study of 48 cavities of edges 48 to 160, launch shape tuned
        dict(name="ensemble_48", kind="ensemble", n=48, draw=2016, sizes="48,64,96,128,160", cubes=True,
             precision=FP32, tune=True, height=0.4, steps=24),
        # a small sweep of odd cavities with FP16 storage, default launch shape
        dict(name="sweep_8_fp16", kind="ensemble", n=8, draw=7, sizes="20,25,33,40,47", cubes=False, precision=FP16,
             tune=False, height=0.4, steps=16),
        # the adjoint: gradient of a front mismatch at 96^3 over the first 1000 steps of a melt
        dict(name="gradient_96", kind="gradient", nx=96, ny=96, nz=96, face=SIDE, Ra=1e5, Pr=0.02, Ste=0.1, Ma=0.1,
             s0=1.0, steps=1000),
        # fields and diagnostics of a large state
        dict(name="readout_256", kind="readout", nx=256, ny=256, nz=256, face=SIDE, precision=FP32, Tc=0.0,
             height=0.4, **convection),
    ]


def draw(rng):
    def edge(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    kind = rng.choice(["melt", "melt", "melt", "subcooled", "loop", "ensemble", "gradient", "readout"])
    Ra = 10 ** rng.uniform(4, 6)
    Pr = 10 ** rng.uniform(math.log10(0.02), 0)
    flow = dict(face=rng.choice([SIDE, BOTTOM]), Ra=Ra, Pr=Pr, Ste=rng.uniform(0.05, 0.2), Ma=0.1)
    box = dict(nx=edge(20, 256), ny=edge(20, 256), nz=edge(20, 256))
    if rng.random() < 0.5:
        box = dict(nx=box["nx"], ny=box["nx"], nz=box["nx"])
    if kind == "ensemble":
        n = rng.randint(2, 24)
        odd = rng.random() < 0.5
        return dict(kind="ensemble", n=n, draw=rng.randint(0, 9999), precision=rng.choice([FP32, FP32, FP16]),
                    sizes="20,25,33,40,47,64,81" if odd else "48,64,96,128", cubes=not odd,
                    tune=rng.random() < 0.5, height=rng.uniform(0.2, 0.6), steps=rng.randint(6, 16))
    if kind == "gradient":
        e = edge(16, 80)
        return dict(kind="gradient", nx=e, ny=edge(16, 80), nz=edge(16, 80), s0=rng.uniform(1.0, 4.0),
                    steps=rng.randint(60, 400), **dict(flow, Pr=rng.uniform(0.02, 0.3)))
    precision = rng.choice([FP32, FP16])
    if kind == "subcooled":
        return dict(kind="melt", precision=FP32, Tc=-rng.uniform(0.05, 0.3), height=rng.uniform(0.1, 0.8),
                    steps=rng.randint(4, 20), restore=True, **box, **flow)
    if kind == "melt":
        return dict(kind="melt", precision=precision, Tc=0.0, height=rng.uniform(0.05, 0.9),
                    steps=rng.randint(4, 8) if precision == FP16 else rng.randint(4, 30), restore=True, **box, **flow)
    if kind == "loop":
        return dict(kind="loop", precision=FP32, Tc=0.0, height=rng.uniform(0.1, 0.8), steps=rng.randint(2, 16),
                    **box, **flow)
    return dict(kind="readout", precision=precision, Tc=0.0, height=rng.uniform(0.1, 0.8), **box, **flow)


# ---------------------------------------------------------------- inputs

def cavity_args(case):
    """The arguments of one cavity's create."""
    H = case["ny"] if case["face"] == SIDE else case["nz"]
    kw = dict(face=case["face"], precision=case.get("precision", FP32), Ra=case["Ra"], Pr=case["Pr"],
              Ste=case["Ste"], Ma=case["Ma"], s0=case.get("s0") or max(1.0, case["height"] * H))
    if case["Ra"] > 0.0:
        kw["derive"] = True
    else:  # conduction with thermal diffusivity 1/4 and viscosity Pr / 4
        kw["s_nu"] = 1.0 / (0.75 * case["Pr"] + 0.5)
        kw["s_alpha"] = 2.0 / 3.0
    if case.get("Tc", 0.0) < 0.0:
        kw.update(Tc=case["Tc"], Tm=0.0, solid=1, ks_kl=1.0)
    return (case["nx"], case["ny"], case["nz"]), kw


def modes(gen, n1, n2, dev):
    """A smooth random field over a plane of n1 x n2, within [-1, 1]."""
    a = (torch.arange(n1, device=dev) + 0.5) / n1
    b = (torch.arange(n2, device=dev) + 0.5) / n2
    c = torch.rand(3, 3, generator=gen, device=dev) * 2 - 1
    out = torch.zeros(n1, n2, device=dev)
    for i in range(3):
        for j in range(3):
            out += c[i, j] * torch.cos(math.pi * (i + 1) * a)[:, None] * torch.cos(math.pi * (j + 1) * b)[None, :] / 9
    return out


def fields(case, seed):
    """A melting state in its natural form: distributions f (19, N) and g (7,
    N) in float32 at the local equilibrium of a convecting liquid under a
    wavy front, the front S (float64) and the heated-wall field."""
    nx, ny, nz, face = case["nx"], case["ny"], case["nz"], case["face"]
    dev = torch.device("cuda")
    gen = torch.Generator(dev).manual_seed(seed)
    H, n1 = (ny, nz) if face == SIDE else (nz, ny)
    s0 = max(1.0, case["height"] * H)
    S = (s0 * (1 + 0.15 * modes(gen, n1, nx, dev))).clamp(0.6, H - 0.1)
    ax = 1 if face == SIDE else 0
    shape = [1, 1, 1]
    shape[ax] = H
    a = (torch.arange(H, device=dev) + 0.5).reshape(shape)
    s3 = S.unsqueeze(ax)
    liq = a < s3
    zeta = (a / s3).clamp(max=1.0)
    bump = torch.sin(math.pi * zeta)
    Tc = case.get("Tc", 0.0)
    T = torch.where(liq, 1.0 - zeta + 0.2 * bump * modes(gen, n1, nx, dev).unsqueeze(ax),
                    Tc * ((a - s3) / (H - s3)).clamp(0.0, 1.0))
    u = [0.1 * bump * modes(gen, n1, nx, dev).unsqueeze(ax) for _ in range(3)]
    rho = 1.0 + 1e-3 * (0.5 + 0.5 * modes(gen, n1, nx, dev).unsqueeze(ax)).expand(nz, ny, nx)
    uu = u[0] ** 2 + u[1] ** 2 + u[2] ** 2
    f = torch.empty(19, nz, ny, nx, device=dev)
    g = torch.empty(7, nz, ny, nx, device=dev)
    for i, e in enumerate(E19):
        eu = e[0] * u[0] + e[1] * u[1] + e[2] * u[2]
        f[i] = torch.where(liq, W19[i] * (rho + 3 * eu + 4.5 * eu * eu - 1.5 * uu), torch.zeros_like(uu))
    for i, e in enumerate(E7):
        eu = e[0] * u[0] + e[1] * u[1] + e[2] * u[2]
        g[i] = torch.where(liq, W7[i] * T * (1 + 4 * eu), W7[i] * T)
    wall = 1.0 + 0.01 * torch.randn(n1, nx, generator=gen, device=dev)
    return f, g, S.double().contiguous(), wall.contiguous()


def members(case):
    """The cavities of an ensemble as melt cases."""
    sizes = tuple(int(v) for v in case["sizes"].split(","))
    drawn = inputs.ensemble(case["n"], case["draw"], sizes=sizes)
    r = random.Random(case["draw"])
    out = []
    for d in drawn:
        box = [d["n"]] * 3 if case["cubes"] else [r.choice(sizes) for _ in range(3)]
        out.append(dict(nx=box[0], ny=box[1], nz=box[2], face=d["face"], precision=case["precision"], Ra=d["Ra"],
                        Pr=0.02, Ste=d["Ste"], Ma=0.1, Tc=0.0, height=case["height"]))
    return out


def pointer(t):
    return ctypes.c_void_p(t.data_ptr())


def restore(cav, saved):
    """Uploads a saved state from device memory (lbm_melt_set_state)."""
    cav._check(_abi.load().lbm_melt_set_state(cav._h, *(pointer(t) for t in saved), 1))


def save(cav, f, g):
    """The state into device memory (lbm_melt_get_state)."""
    cav._check(_abi.load().lbm_melt_get_state(cav._h, pointer(f), pointer(g), None, 1))


def outputs_of(case):
    shape = (case["nz"], case["ny"], case["nx"])
    cols = (case["nz"] if case["face"] == SIDE else case["ny"], case["nx"])
    return dict(T=torch.empty(shape, device="cuda"), u=torch.empty(shape + (3,), device="cuda"),
                S=torch.empty(cols, dtype=torch.float64, device="cuda"),
                lf=torch.empty(1, dtype=torch.float64, device="cuda"))


def target(case, seed):
    n1 = case["nz"] if case["face"] == SIDE else case["ny"]
    gen = torch.Generator("cuda").manual_seed(seed)
    dTh = 0.01 * torch.randn(n1, case["nx"], generator=gen, device="cuda")
    return dTh, case["s0"] + 2.0 + modes(gen, n1, case["nx"], torch.device("cuda"))


def prepare(case, seed):
    if case["kind"] == "gradient":
        dTh, goal = target(case, seed)
        spec = dict(nx=case["nx"], ny=case["ny"], nz=case["nz"], face=case["face"], Pr=case["Pr"], Ste=case["Ste"],
                    Ma=case["Ma"], s0=case["s0"])
        return dict(case=case, dTh=dTh.requires_grad_(), Ra=torch.tensor(case["Ra"], requires_grad=True), goal=goal,
                    spec=spec)
    if case["kind"] == "ensemble":
        cases = members(case)
        args = []
        for c in cases:
            (nx, ny, nz), kw = cavity_args(c)
            args.append(dict(nx=nx, ny=ny, nz=nz, **kw))
        ens = Ensemble(args)
        if case["tune"]:
            autotune.tune_ensemble(ens)
        cavs = [ens.member(i) for i in range(ens.n)]
        saved = []
        for i, c in enumerate(cases):
            f, g, S, wall = fields(c, seed * 64 + i)
            cavs[i].set_hot_wall(wall)
            saved.append((f, g, S))
        return dict(case=case, ens=ens, cavs=cavs, saved=saved, out=[outputs_of(c) for c in cases])
    dims, kw = cavity_args(case)
    cav = Cavity(*dims, **kw)
    f, g, S, wall = fields(case, seed)
    if case["kind"] != "readout":  # there the wall stays at Th
        cav.set_hot_wall(wall)
    restore(cav, (f, g, S))
    state = dict(case=case, cav=cav, out=outputs_of(case))
    if case.get("restore"):
        state["saved"] = (f, g, S)
        state["end"] = (torch.empty_like(f), torch.empty_like(g))
    if case["kind"] == "loop":
        state["walls"] = [(wall * (1.0 + 0.002 * k)).cpu().pin_memory() for k in range(4)]
        state["S"] = torch.empty((case["steps"],) + tuple(S.shape), dtype=torch.float64).pin_memory()
        state["lf"] = torch.empty(case["steps"], dtype=torch.float64).pin_memory()
    return state


def run(state):
    case = state["case"]
    if case["kind"] == "melt":
        cav, out = state["cav"], state["out"]
        if "saved" in state:
            restore(cav, state["saved"])
        cav.step(case["steps"])
        cav.get_device(**out)
        if "saved" in state:
            save(cav, *state["end"])
            return dict(out, f=state["end"][0], g=state["end"][1])
        return out
    if case["kind"] == "ensemble":
        for cav, saved in zip(state["cavs"], state["saved"]):
            restore(cav, saved)
        state["ens"].step(case["steps"])
        for cav, out in zip(state["cavs"], state["out"]):
            cav.get_device(**out)
        if len(state["out"]) <= 12:
            return state["out"]
        return {k: torch.cat([o[k].reshape(-1) for o in state["out"]]) for k in ("T", "u", "S", "lf")}
    if case["kind"] == "gradient":
        # parameters, front and loss in float32, as a torch optimiser holds them
        state["dTh"].grad = state["Ra"].grad = None
        S = melt_front(state["dTh"], state["Ra"], state["spec"], case["steps"]).float()
        loss = ((S - state["goal"]) ** 2).mean()
        loss.backward()
        return dict(S=S.detach(), loss=loss.detach(), dTh=state["dTh"].grad, Ra=state["Ra"].grad)
    if case["kind"] == "loop":
        cav, L = state["cav"], _abi.load()
        for k in range(case["steps"]):
            cav._check(L.lbm_melt_set_hot_wall(cav._h, pointer(state["walls"][k % 4]), 0))
            cav.step(1)
            cav._check(L.lbm_melt_get_async(cav._h, pointer(state["S"][k]), pointer(state["lf"][k]), 0))
        cav.get_device(T=state["out"]["T"])  # waits for the copies too
        return dict(S=state["S"], lf=state["lf"], T=state["out"]["T"])
    cav, out = state["cav"], state["out"]
    cav.get_device(**out)
    nu, mean = cav.nusselt()
    return dict(out, totals=cav.totals(), nusselt=nu, nusselt_mean=mean)


# ------------------------------------------------------------------ work

FLOP_LIQUID, FLOP_SOLID = 420, 60  # of one collision (19 + 7 moments, their equilibria, and back), of a solid node's


def work(case):
    """Bytes and operations of a pass: a step reads and writes every liquid
    node's 26 populations (and a conducting solid node's 7), a pass its
    state, walls and outputs."""
    if case["kind"] == "ensemble":
        parts = [work(dict(c, kind="melt", steps=case["steps"], restore=True, member=True)) for c in members(case)]
        return {k: sum(p[k] for p in parts) for k in ("bytes", "flops")}
    N = case["nx"] * case["ny"] * case["nz"]
    H = case["ny"] if case["face"] == SIDE else case["nz"]
    cols = N // H
    if case["kind"] == "gradient":
        # forward, recomputation and reverse sweep (which reads the state and the adjoint and writes the
        # adjoint); the layer grows as sqrt(s0^2 + 2 alpha Ste t)
        alpha = case["Ma"] / math.sqrt(3) * H * math.sqrt(case["Pr"] / case["Ra"]) / case["Pr"]
        s = sum(math.sqrt(case["s0"] ** 2 + 2 * alpha * case["Ste"] * t) for t in range(case["steps"]))
        nodes = min(s, H * case["steps"]) * cols
        return {"bytes": nodes * (208 + 208 + 312), "flops": nodes * 4 * FLOP_LIQUID}
    es = 2 if case["precision"] == FP16 else 4
    liquid = min(max(1.0, case["height"] * H), H) * cols
    conducting = N - liquid if case.get("Tc", 0.0) < 0.0 else 0
    steps = case.get("steps", 0)
    b = steps * (liquid * 52 * es + conducting * 14 * es + cols * 2 * 8)
    fl = steps * (liquid * FLOP_LIQUID + conducting * FLOP_SOLID)
    if case["kind"] == "loop":
        return {"bytes": b + steps * cols * 12 + N * 4 + liquid * 7 * es, "flops": fl}
    b += N * 16 + liquid * 26 * es + cols * 8  # the fields out
    if case.get("restore"):
        b += (liquid * 26 + conducting * 7) * (4 + es) + cols * 8
        b += 0 if case.get("member") else N * 26 * 4 + (liquid * 26 + conducting * 7) * es
    if case["kind"] == "readout":
        b += cols * 8
    return {"bytes": b, "flops": fl + liquid * 60}


# ----------------------------------------------------------------- exact
# The method in 64 bits: two copies of the state, pull streaming, matrices
# for the moments, every rule a masked tensor expression, so that torch can
# also differentiate it (phase flags held at their forward values).

def polynomials():
    M, N = [], []
    for x, y, z in E19:
        q = x * x + y * y + z * z
        M.append([1, 19 * q - 30, (21 * q * q - 53 * q + 24) // 2, x, (5 * q - 9) * x, y, (5 * q - 9) * y, z,
                  (5 * q - 9) * z, 3 * x * x - q, (3 * q - 5) * (3 * x * x - q), y * y - z * z,
                  (3 * q - 5) * (y * y - z * z), x * y, y * z, x * z, (y * y - z * z) * x, (z * z - x * x) * y,
                  (x * x - y * y) * z])
    for x, y, z in E7:
        q = x * x + y * y + z * z
        N.append([1, x, y, z, 6 - 7 * q, 3 * x * x - q, y * y - z * z])
    return (torch.tensor(M, dtype=torch.float64).T.contiguous().cuda(),
            torch.tensor(N, dtype=torch.float64).T.contiguous().cuda())


class Exact:
    """One cavity in 64 bits; `top` cuts the heating axis above the liquid
    (solid at Tm = 0 there, which nothing changes)."""

    def __init__(self, case, wall, top=None, Ra=None):
        self.face, self.conduct = case["face"], case.get("Tc", 0.0) < 0.0
        self.H = case["ny"] if case["face"] == SIDE else case["nz"]
        self.h = self.H if top is None or self.conduct else min(self.H, top)
        self.Tc, self.wall = case.get("Tc", 0.0), wall
        self.ax = 1 if self.face == SIDE else 0
        self.dims = [case["nz"], case["ny"], case["nx"]]
        self.dims[self.ax] = self.h
        shape = [1, 1, 1]
        shape[self.ax] = self.h
        self.a = torch.arange(self.h, device="cuda").reshape(shape)
        if case["Ra"] > 0.0:
            Ra = torch.tensor(case["Ra"], dtype=torch.float64, device="cuda") if Ra is None else Ra
            nu = case["Ma"] / math.sqrt(3) * self.H * torch.sqrt(case["Pr"] / Ra)
            alpha = nu / case["Pr"]
            self.gb = Ra * nu * alpha / self.H ** 3
        else:
            nu = torch.tensor(0.25 * case["Pr"], dtype=torch.float64, device="cuda")
            alpha, self.gb = torch.full_like(nu, 0.25), torch.zeros_like(nu)
        self.alpha, self.coef = alpha, alpha * case["Ste"]
        M, N = polynomials()
        Mi, Ni = torch.linalg.inv(M), torch.linalg.inv(N)
        one = torch.ones_like(alpha)
        sn, sa = 1 / (3 * nu + 0.5), 1 / (4 * alpha + 0.5)
        rates = [1.0, 1.19, 1.4, 1.0, 1.2, 1.0, 1.2, 1.0, 1.2, sn, 1.4, sn, 1.4, sn, sn, sn, 1.98, 1.98, 1.98]
        R = torch.stack([one * r for r in rates])
        Q = torch.stack([one * r for r in [1.0, sa, sa, sa, 1.0, 1.0, 1.0]])
        self.A = Mi @ (R[:, None] * M)                # f* = f - A (f - feq) + B F
        self.B = Mi @ ((1 - 0.5 * R)[:, None] * M)
        self.C = Ni @ (Q[:, None] * N)                # g* = g - C (g - geq); k_s = k_l: the solid's too
        self.e = torch.tensor(E19, dtype=torch.float64, device="cuda")
        self.inside = [self._inside(d) for d in E19]

    def _inside(self, d):
        m = torch.ones(self.dims, dtype=torch.bool, device="cuda")
        for ax, v in ((2, d[0]), (1, d[1]), (0, d[2])):
            if v:
                m.narrow(ax, 0 if v > 0 else self.dims[ax] - 1, 1).fill_(False)
        return m

    def col(self, c):  # a per-column field against the nodes
        return c.unsqueeze(self.ax)

    def at(self, field, j):  # the field's value at height j of each column
        return torch.gather(field, self.ax, self.col(j.clamp(0, self.h - 1))).squeeze(self.ax)

    def upstream(self, x, d):
        return torch.roll(x, (d[2], d[1], d[0]), (0, 1, 2)) if any(d) else x

    def counts(self, s):
        return torch.ceil(s.detach() - 0.5).clamp(0, self.H).long()

    def geq(self, T, u):
        return torch.stack([W7[i] * T * (1 + 4 * (e[0] * u[0] + e[1] * u[1] + e[2] * u[2])) for i, e in enumerate(E7)])

    def velocity(self, f, T, liq):
        j = (self.e.T @ f.reshape(19, -1)).reshape([3] + self.dims)
        zero = torch.zeros_like(T)
        F = self.gb * T
        return [torch.where(liq, v, zero) for v in (j[0], j[1], j[2] + 0.5 * F)], F

    def collide_g(self, g, T, u):
        shape = g.shape
        return g - (self.C @ (g - self.geq(T, u)).reshape(7, -1)).reshape(shape)

    def ghosts(self, f, g, s, js, wall):
        """Post-collision populations of each column's ghost nodes: of the
        first solid node, and of the last liquid one towards the solid."""
        T = g.sum(0)
        liq = self.a < self.col(js)
        k = torch.floor(s.detach() - 1).long().clamp(max=self.H - 1)
        yg = js + 0.5
        Tk = self.at(T, k)
        near = -wall * (yg - s) / s
        line = -Tk * (yg - s) / (s - (k + 0.5))
        Tg = torch.where(k < 0, near, line)

        def with_rest(Tghost, j, u):
            TL = self.at(T, j)
            gL = torch.stack([self.at(x, j) for x in g])
            uL = [self.at(x, j) for x in u]
            eq = self.geq(TL, uL)
            neq = (gL - eq) - (self.C @ (gL - eq).reshape(7, -1)).reshape(gL.shape)
            both = (js >= 1) & (js < self.H)
            rest = torch.stack([w * Tghost for w in W7])
            return rest + torch.where(both, neq, torch.zeros_like(neq))

        u, _ = self.velocity(f, T, liq)
        liquid_side = with_rest(Tg, js - 1, u)
        if not self.conduct:
            return liquid_side, None
        ks = torch.ceil(s).long()
        ys = js - 0.5
        Ts = torch.where(ks >= self.H, self.Tc * (ys - s) / (self.H - s).clamp(min=1e-9),
                         self.at(T, ks) * (ys - s) / ((ks + 0.5) - s))
        Ts = torch.where((js < 1) | (js >= self.H), torch.zeros_like(Ts), Ts)
        return liquid_side, with_rest(Ts, js, [torch.zeros_like(T)] * 3)

    def step(self, f, g, s, js, ghost, wall):
        a, H = self.a, self.H
        liq = a < self.col(js)
        T = g.sum(0)
        u, F = self.velocity(f, T, liq)
        uu = u[0] ** 2 + u[1] ** 2 + u[2] ** 2
        rho = f.sum(0)
        feq, force = [], []
        for i, e in enumerate(E19):
            eu = e[0] * u[0] + e[1] * u[1] + e[2] * u[2]
            feq.append(W19[i] * (rho + 3 * eu + 4.5 * eu * eu - 1.5 * uu))
            force.append(W19[i] * (3 * (e[2] - u[2]) + 9 * eu * e[2]) * F)
        fs = f - (self.A @ (f - torch.stack(feq)).reshape(19, -1)).reshape(f.shape)
        fs = fs + (self.B @ torch.stack(force).reshape(19, -1)).reshape(f.shape)
        del feq, force
        gs = self.collide_g(g, T, u)
        is_ghost = a == self.col(js)
        front = torch.stack([self.col(x).expand(self.dims) for x in ghost[0]])
        zero = torch.zeros_like(gs)
        if self.conduct:
            last = a == self.col(js) - 1
            back = torch.stack([self.col(x).expand(self.dims) for x in ghost[1]])
            cross = torch.where(liq, torch.where(last, back, zero), torch.where(is_ghost, front, zero))
        else:
            gs = torch.where(liq, gs, torch.where(is_ghost, front, zero))
        fn = [fs[0]]
        for i in range(1, 19):
            from_liquid = self.upstream(liq, E19[i]) & self.inside[i]
            fn.append(torch.where(from_liquid, self.upstream(fs[i], E19[i]), fs[OPP19[i]]))
        f = torch.where(liq, torch.stack(fn), torch.zeros_like(fs))
        del fn, fs
        gn = [gs[0]]
        for i in range(1, 7):
            v = self.upstream(gs[i], E7[i])
            if self.conduct:
                v = torch.where(self.upstream(liq, E7[i]) == liq, v, self.upstream(cross[i], E7[i]))
            out = gs[OPP7[i]]
            d = E7[i][1] if self.face == SIDE else E7[i][2]
            if d:
                out = -out + 2 * W7[i] * (self.col(wall) if d > 0 else self.Tc)
            gn.append(torch.where(self.inside[i], v, out))
        g = torch.stack(gn)
        # the front: Eq. 6 with central slopes, mirrored at the side walls
        T = g.sum(0)
        k = torch.floor(s.detach() - 1).long().clamp(max=H - 1)
        y1, y0 = self.at(T, k), torch.where(k >= 1, self.at(T, k - 1), wall)
        x1 = k + 0.5
        x0 = torch.where(k >= 1, k - 0.5, torch.zeros_like(x1))
        quad = y0 * (s - x1) / ((x0 - x1) * (x0 - s)) + y1 * (s - x0) / ((x1 - x0) * (x1 - s))
        G = torch.where(k < 0, -wall / s, quad)
        if self.conduct:
            ks = torch.ceil(s).long()
            z1, z2 = ks + 0.5, torch.where(ks + 1 < H, ks + 1.5, torch.full_like(s, float(H)))
            Y2 = torch.where(ks + 1 < H, self.at(T, ks + 1), torch.full_like(s, self.Tc))
            Gs = self.at(T, ks) * (s - z2) / ((z1 - s) * (z1 - z2)) + Y2 * (s - z1) / ((z2 - s) * (z2 - z1))
            Gs = torch.where(ks >= H, self.Tc / (H - s).clamp(min=1e-9), Gs)
            G = G - torch.where(js < H, Gs, torch.zeros_like(Gs))
        sp = 0.5 * (torch.cat([s[:, 1:], s[:, -1:]], 1) - torch.cat([s[:, :1], s[:, :-1]], 1))
        sq = 0.5 * (torch.cat([s[1:], s[-1:]], 0) - torch.cat([s[:1], s[:-1]], 0))
        s = (s + self.coef * (1 + sp ** 2 + sq ** 2) * (-G)).clamp(0.5, float(H))
        new = self.counts(s)
        now = a < self.col(new)
        rest = torch.tensor(W19, dtype=torch.float64, device="cuda").reshape(19, 1, 1, 1)
        f = torch.where(now & ~liq, rest, torch.where(now, f, torch.zeros_like(f)))
        return f, g, s, new, self.ghosts(f, g, s, new, wall)

    def start(self, f, g, S):
        s = S.double()
        js = self.counts(s)
        liq = self.a < self.col(js)
        f = torch.where(liq, f.narrow(1 + self.ax, 0, self.h).double(), torch.zeros((), dtype=torch.float64, device="cuda"))
        g = g.narrow(1 + self.ax, 0, self.h).double()
        if not self.conduct:
            g = torch.where(liq, g, torch.zeros((), dtype=torch.float64, device="cuda"))
        return f, g, s, js, self.ghosts(f, g, s, js, self.wall)

    def macro(self, f, g, s, js, ghost=None):
        liq = self.a < self.col(js)
        T = g.sum(0)
        u, _ = self.velocity(f, T, liq)
        T = T if self.conduct else torch.where(liq, T, torch.zeros_like(T))
        u = torch.stack(u, -1)
        return dict(T=self.whole(T), u=self.whole(u), S=s, lf=(s.sum() / (self.H * s.numel())).reshape(1))

    def whole(self, x, lead=0):  # zeros above the cut
        if self.h == self.H:
            return x
        more = list(x.shape)
        more[lead + self.ax] = self.H - self.h
        return torch.cat([x, x.new_zeros(more)], lead + self.ax)

    def initial(self, case):
        """The library's own start: a flat front over the Neumann profile."""
        lo, hi = 0.0, 2.0
        for _ in range(200):
            mid = 0.5 * (lo + hi)
            lo, hi = (mid, hi) if mid * math.exp(mid * mid) * math.erf(mid) < case["Ste"] / math.sqrt(math.pi) else (lo, mid)
        prof = [1 - math.erf((j + 0.5) * lo / case["s0"]) / math.erf(lo) if j + 0.5 < case["s0"] else 0.0 for j in range(self.h)]
        T = torch.tensor(prof, dtype=torch.float64, device="cuda").reshape(self.a.shape).expand(self.dims)
        g = torch.stack([w * T for w in W7])
        cols = [d for k, d in enumerate(self.dims) if k != self.ax]
        s = torch.full(cols, case["s0"], dtype=torch.float64, device="cuda")
        js = self.counts(s)
        f = torch.stack([w * (self.a < self.col(js)).double().expand(self.dims) for w in W19])
        return f, g, s, js, self.ghosts(f, g, s, js, torch.ones_like(s))


def exact_melt(case, seed):
    f, g, S, wall = fields(case, seed)
    wall = torch.ones_like(wall) if case["kind"] == "readout" else wall
    ref = Exact(case, wall.double(), top=int(S.max()) + 8)
    st = ref.start(f, g, S)
    del f, g
    for _ in range(case.get("steps", 0)):
        st = ref.step(*st, ref.wall)
    return ref, st


def exact_gradient(case, seed):
    dTh, goal = target(case, seed)
    Ra = torch.tensor(case["Ra"], dtype=torch.float64, device="cuda", requires_grad=True)
    wall = (1.0 + dTh.double()).float().double().requires_grad_()
    H = case["ny"] if case["face"] == SIDE else case["nz"]
    alpha = case["Ma"] / math.sqrt(3) * H * math.sqrt(case["Pr"] / case["Ra"]) / case["Pr"]
    top = int(1.5 * math.sqrt(case["s0"] ** 2 + 2 * alpha * case["Ste"] * case["steps"])) + 8
    ref = Exact(case, wall, top=top, Ra=Ra)
    f, g, s, js, ghost = ref.initial(case)
    from torch.utils.checkpoint import checkpoint

    def piece(f, g, s, gh, w, js):
        f, g, s, js, ghost = ref.step(f, g, s, js, (gh, None), w)
        return f, g, s, js, ghost[0]

    gh = ghost[0]
    for _ in range(case["steps"]):
        f, g, s, js, gh = checkpoint(piece, f, g, s, gh, wall, js, use_reentrant=False)
    loss = ((s - goal.double()) ** 2).mean()
    gw, gr = torch.autograd.grad(loss, [wall, Ra])
    return dict(S=s.detach(), loss=loss.detach(), dTh=gw, Ra=gr)


def exact(case, seed):
    if case["kind"] == "gradient":
        return exact_gradient(case, seed)
    if case["kind"] == "ensemble":
        out = []
        for i, c in enumerate(members(case)):
            ref, st = exact_melt(dict(c, kind="melt", steps=case["steps"]), seed * 64 + i)
            out.append(ref.macro(*st))
        if len(out) <= 12:
            return out
        return {k: torch.cat([o[k].reshape(-1) for o in out]) for k in ("T", "u", "S", "lf")}
    if case["kind"] == "melt":
        ref, st = exact_melt(case, seed)
        out = ref.macro(*st)
        return dict(out, f=ref.whole(st[0], 1), g=ref.whole(st[1], 1)) if case["restore"] else out
    if case["kind"] == "loop":
        f, g, S, wall = fields(case, seed)
        ref = Exact(case, wall.double(), top=int(S.max()) + 8)
        st = ref.start(f, g, S)
        Ss = []
        for k in range(case["steps"]):
            w = (wall * (1.0 + 0.002 * (k % 4))).double()
            st = ref.step(*st, w)
            Ss.append(st[2].cpu())
        out = ref.macro(*st)
        Ss = torch.stack(Ss)
        return dict(S=Ss, lf=Ss.mean((1, 2)) / ref.H, T=out["T"])
    ref, st = exact_melt(case, seed)
    f, g, s, js, _ = st
    out = ref.macro(*st)
    liq = ref.a < ref.col(js)
    # heat through the heated-wall link: the node's incoming population is given, -g_out + 2 w Tw = g_in
    up = 3 if case["face"] == SIDE else 5
    q = 2 * (g[up].select(ref.ax, 0) - W7[up] * ref.wall)
    nu = q * ref.H / ref.alpha
    speed = (out["u"] ** 2).sum(-1).max().sqrt()
    totals = dict(liquid_fraction=float(out["lf"]), sum_T_minus_Tm=float(out["T"].sum()),
                  sum_rho_minus_1=float(torch.where(liq, f.sum(0) - 1, torch.zeros_like(g[0])).sum()),
                  n_liquid=float(js.sum()), max_u=float(speed), sum_S=float(s.sum()), nusselt_mean=float(nu.mean()))
    return dict(out, totals=totals, nusselt=nu.cpu().numpy(), nusselt_mean=float(nu.mean()))
