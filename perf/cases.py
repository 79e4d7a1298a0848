"""Workloads that stand for what a user of this library has it do, each through
its public entry points, with an independent FP64 statement of the result.

Kinds of case:
  step      advance one simulation by some steps, then read its macroscopic
            fields on the device (the inner loop of every study);
  batch     one tick of the serving loop: many resident simulations advanced
            together, then their conversion polled and species read;
  poll      the observables of a running simulation (profiles and site map);
  snapshot  every macroscopic field of a running simulation;
  sample    a new request: synthetic sample, simulation, first fields.

Samples: a thresholded smooth random field with the porosity and correlation
length given, handed over as a caller mask ("field"), pore disks carved out of
a thin ingot ("disks"), two parallel plates ("plates"), or the library's own
generator ("generated", in the cases of kind sample).
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_1607_02874_gb300 import lbm

STORAGE = {"fp32": lbm.FP32, "fp16": lbm.FP16_DEV, "bf16": lbm.BF16_DEV}
LAYOUT = {"auto": lbm.LAYOUT_AUTO, "dense": lbm.LAYOUT_DENSE, "fluid": lbm.LAYOUT_FLUID}

# What a case leaves out. u_in < 0: the pressure inlet; p < 0: from Da.
DEFAULTS = dict(kind="step", sample="field", storage="fp32", layout="auto", n_species=2, steps=1, corr_len=6.0,
                porosity=0.65, Da=1.0, p=-1.0, tau=0.8, tau_s=0.0, g_z=0.0, rho_in=1.001, rho_out=1.0, c_in=1.0,
                c_init=1.0, pS_R=0.95, pS_P=0.0, u_in=-1.0, bary=False, random=False, desorb=False,
                deterministic=False, count=1, side_lo=0, side_hi=0, thickness=0)


def _box(nx, ny, nz, z0, z1, **kw):
    return dict(DEFAULTS, nx=nx, ny=ny, nz=nz, z0=z0, z1=z1, **kw)


def listed():
    return [
        # The plain method on its smallest box (carrier and reactant): what a
        # first run and every quick check cost, all launches and latency.
        _box(32, 32, 64, 16, 48, name="small_32x32x64_cr_fp32", n_species=1, steps=200),
        # The validation channel: thin box, inert and reactive plates, a body
        # force and a species relaxation time of their own.
        _box(52, 1, 154, 2, 152, name="channel_52x1x154_fp32", sample="plates", tau=1.0, tau_s=0.55, g_z=4.5e-5,
             rho_in=1.0, p=1.0, pS_R=1.0, steps=300),
        # The two-dimensional reactor with the paper's own ingot: barycentric
        # velocity, velocity inlet, thin box.
        _box(500, 1, 250, 120, 130, name="reactor_500x1x250_bary_fp32", sample="disks", porosity=0.70, thickness=200,
             tau=4.0, rho_in=0.8, rho_out=0.8, c_in=0.2, c_init=0.2, u_in=0.08, p=0.45, bary=True, steps=300),
        # A ragged box with the random sputtering matrix in dense addressing,
        # an odd number of steps.
        _box(37, 29, 50, 12, 38, name="ragged_37x29x50_random_bf16", storage="bf16", layout="dense", corr_len=3.0,
             porosity=0.6, random=True, p=0.45, pS_P=0.1, steps=101),
        # One point of the Damkohler-number sweep.
        _box(128, 128, 256, 64, 192, name="sweep_128x128x256_fp16", storage="fp16", porosity=0.60, corr_len=10.0,
             Da=0.1, steps=100),
        # The precision study's sample, in FP32.
        _box(256, 256, 512, 128, 384, name="sample_256x256x512_fp32", porosity=0.70, corr_len=14.0, steps=24),
        # A sample of odd sizes filled with solid nearly from end to end, in
        # bfloat16, an odd number of steps.
        _box(191, 173, 300, 6, 294, name="porous_191x173x300_bf16", storage="bf16", porosity=0.62, corr_len=8.0,
             desorb=True, steps=41),
        # The largest sample, in FP16.
        _box(512, 512, 1024, 128, 896, name="sample_512x512x1024_fp16", storage="fp16", corr_len=20.0, Da=0.1,
             steps=50),
        # One tick of the serving loop: boxes of side 48 to 192.
        dict(DEFAULTS, name="serving_24_fp16", kind="batch", storage="fp16", layout="fluid", count=24, side_lo=48,
             side_hi=192, deterministic=True, steps=40),
        # Polling a running simulation: conversion, profiles, site map.
        _box(256, 256, 512, 128, 384, name="poll_256x256x512_fp16", kind="poll", storage="fp16", porosity=0.70,
             corr_len=14.0, steps=10),
        # Reading every field of a running simulation, at an odd step.
        _box(256, 256, 512, 128, 384, name="snapshot_256x256x512_fp32", kind="snapshot", porosity=0.70,
             corr_len=14.0, steps=11),
        # A new request: generate the sample, start the simulation, first look.
        _box(128, 128, 256, 64, 192, name="new_sample_128x128x256_fp16", kind="sample", sample="generated",
             storage="fp16", porosity=0.60, corr_len=10.0, Da=0.1),
    ]


def draw(rng):
    kind = rng.choices(("step", "batch", "poll", "snapshot", "sample"), (12, 2, 2, 2, 2))[0]
    c = dict(DEFAULTS, kind=kind, storage=rng.choice(("fp32", "fp16", "bf16")), n_species=rng.choice((1, 2, 2)),
             porosity=rng.uniform(0.55, 0.75), corr_len=rng.uniform(3.0, 16.0), Da=10 ** rng.uniform(-3, 1),
             deterministic=rng.random() < 0.25)
    if kind == "batch":
        lo = rng.randint(32, 120)
        c.update(layout="fluid", n_species=2, deterministic=True, count=rng.randint(3, 28), side_lo=lo,
                 side_hi=rng.randint(lo + 1, 192), steps=rng.randint(7, 60), storage=rng.choice(("fp32", "fp16")))
        return c
    top = {"step": 26.5, "poll": 25.0, "snapshot": 25.0, "sample": 23.5}[kind]
    cells = 2.0 ** rng.uniform(13.0, top)
    nx = max(8, round((cells / 2) ** (1 / 3) * rng.uniform(0.6, 1.5)))
    ny = max(8, round((cells / 2) ** (1 / 3) * rng.uniform(0.6, 1.5)))
    nz = max(16, round(cells / (nx * ny)))
    z0 = rng.randint(2, max(2, nz // 3))
    c.update(nx=nx, ny=ny, nz=nz, z0=z0, z1=rng.randint(max(z0 + 4, nz // 2), nz - 2))
    if kind == "sample":
        c.update(sample="generated", n_species=2)
        return c
    c["steps"] = rng.randint(1, 20) if kind != "step" else max(3, min(200, int(3e9 / (nx * ny * nz)))) - rng.randint(0, 2)
    c["layout"] = rng.choice(("auto", "auto", "auto", "fluid", "dense"))
    option = rng.choice(("none", "none", "none", "none", "random", "bary", "inlet", "desorb", "product"))
    if option == "random":
        c["random"] = True
    elif option == "bary":
        c.update(bary=True, n_species=2, c_in=0.2, c_init=0.2)
    elif option == "inlet":
        c["u_in"] = rng.uniform(0.01, 0.08)
    elif option == "desorb":
        c["desorb"] = True
    elif option == "product":
        c.update(n_species=2, pS_P=rng.uniform(0.05, 0.5), p=rng.uniform(0.1, 0.9))
    return c


# ---- inputs ----------------------------------------------------------------

def _mask(c, seed):
    """[nz, ny, nx] uint8 on the GPU: 0 fluid, 1 catalytic solid, 2 inert."""
    nx, ny, nz, z0, z1 = c["nx"], c["ny"], c["nz"], c["z0"], c["z1"]
    m = torch.zeros((nz, ny, nx), dtype=torch.uint8, device="cuda")
    if c["sample"] == "plates":
        m[z0:z1, :, 0] = 1
        m[z0:z1, :, nx - 1] = 2
        return m
    if c["sample"] == "disks":  # pore disks of diameter 3 carved out of an ingot
        w, x0 = z1 - z0, (nx - c["thickness"]) // 2
        rng = np.random.default_rng(seed)
        ingot = np.ones((w, c["thickness"]), bool)
        z, x = np.mgrid[0:w, 0:c["thickness"]] + 0.5
        while 1.0 - ingot.mean() < c["porosity"]:
            ingot &= (x - rng.uniform(0, c["thickness"])) ** 2 + (z - rng.uniform(0, w)) ** 2 > 2.25
        m[z0:z1, 0, x0:x0 + c["thickness"]] = torch.from_numpy(ingot.astype(np.uint8)).cuda()
        return m
    g = torch.Generator(device="cuda").manual_seed(int(seed))
    v = torch.fft.rfftn(torch.randn((nz, ny, nx), generator=g, device="cuda"))
    for axis, n in enumerate((nz, ny, nx)):  # Gaussian smoothing of covariance exp(-r^2 / 2 l^2)
        k = 2 * math.pi * (torch.fft.rfftfreq(n) if axis == 2 else torch.fft.fftfreq(n)).cuda()
        v *= torch.exp(-0.25 * (k * c["corr_len"]) ** 2).reshape([-1 if a == axis else 1 for a in range(3)])
    v = torch.fft.irfftn(v, s=(nz, ny, nx))[z0:z1]
    cut = v.mean() + v.std() * math.sqrt(2.0) * torch.erfinv(torch.tensor(2 * c["porosity"] - 1.0, device="cuda"))
    m[z0:z1] = (v > cut).to(torch.uint8)
    return m


def _force(c, seed):
    """The body force of this run (the channel is run at several)."""
    return c["g_z"] * np.random.default_rng(seed).uniform(0.7, 1.3) if c["g_z"] else 0.0


def _sides(c):
    """The sides of a batch's boxes, uniform between the smallest and the largest."""
    rng = np.random.default_rng(c["count"])
    return [int(s) for s in rng.integers(c["side_lo"], c["side_hi"] + 1, c["count"])]


def _members(c, seed):
    """The boxes of a batch, each as a case of its own, with its seed."""
    rng = np.random.default_rng(seed)
    out = []
    for side in _sides(c):
        out.append((dict(c, nx=side, ny=side, nz=side, z0=side // 4, z1=3 * side // 4,
                         porosity=float(rng.uniform(0.55, 0.75)), corr_len=float(rng.uniform(4.0, 16.0)),
                         Da=float(10 ** rng.uniform(-3, 1))), int(rng.integers(1 << 30))))
    return out


def _simulate(c, seed, geom):
    return lbm.Simulation(
        geom, tau=c["tau"], rho_in=c["rho_in"], rho_out=c["rho_out"], c_in=c["c_in"], Da=c["Da"],
        p=None if c["p"] < 0 else c["p"], pS_R=c["pS_R"], pS_P=c["pS_P"], n_species=c["n_species"],
        storage=STORAGE[c["storage"]], layout=LAYOUT[c["layout"]], deterministic=c["deterministic"],
        sputter=lbm.SPUTTER_RANDOM if c["random"] else lbm.SPUTTER_UNIFORM, sputter_seed=seed,
        velocity=lbm.VELOCITY_BARYCENTRIC if c["bary"] else lbm.VELOCITY_CARRIER,
        u_in=None if c["u_in"] < 0 else c["u_in"], tau_s=c["tau_s"] or None, g_z=_force(c, seed), desorb=c["desorb"],
        c_init=c["c_init"])


def _polled(c, seed):
    """(case, sample seed) of a polled simulation: one sample, each run at a
    Damkohler number of its own."""
    return dict(c, Da=float(10 ** np.random.default_rng(seed).uniform(-3, 1))), 3


def _generator_seed(seed):
    """Seeds far apart: the generator's noise is the same for seeds that
    differ in the two lowest bits alone."""
    return (seed * 0x9E3779B97F4A7C15) % (1 << 62)


def _build(c, seed):
    geom = lbm.Geometry(c["nx"], c["ny"], c["nz"], slab=(c["z0"], c["z1"]), seed=seed, mask=_mask(c, seed).cpu().numpy())
    return geom, _simulate(c, seed, geom)


def _names(c):
    """The fields that a case of kind step or snapshot reads (not those that
    are zero up to rounding in thin boxes)."""
    if c["sample"] == "plates":
        return ["drho_C", "uz", "rho_R", "rho_P"]
    return ["drho_C", "ux"] + ["uy"] * (c["ny"] > 1) + ["uz", "rho_R"] + ["rho_P"] * (c["n_species"] == 2)


def prepare(case, seed):
    c = dict(case)
    if c["kind"] == "sample":
        n = c["nx"] * c["ny"] * c["nz"]
        return {"c": c, "seed": _generator_seed(seed), "out": {k: torch.empty(n, device="cuda") for k in ("rho_C", "rho_R")}}
    if c["kind"] == "batch":
        boxes = [_build(m, s) for m, s in _members(c, seed)]
        return {"c": c, "boxes": boxes, "out": [{k: torch.empty(g.n, device="cuda") for k in ("rho_R", "rho_P")}
                                                for g, _ in boxes]}
    geom, sim = _build(*_polled(c, seed)) if c["kind"] == "poll" else _build(c, seed)
    if c["kind"] in ("poll", "snapshot"):
        sim.step(c["steps"])
    out = {} if c["kind"] == "poll" else {k: torch.empty(geom.n, device="cuda") for k in _names(c)}
    return {"c": c, "geom": geom, "sim": sim, "out": out}


# (the mass-balance residuals, differences of these down to rounding noise,
# say nothing here)
SCALARS = ("M_C", "M_R", "M_P", "eta", "in_C", "in_R", "out_C", "hits_R", "hits_P", "reacted", "stuck_R", "delta", "p")
PROFILES = ("rhoC_z", "rhoR_z", "rhoP_z", "phiP_z", "react_z")


def run(state):
    c = state["c"]
    if c["kind"] == "sample":
        geom = lbm.Geometry(c["nx"], c["ny"], c["nz"], slab=(c["z0"], c["z1"]), porosity=c["porosity"],
                            corr_len=c["corr_len"], seed=state["seed"])
        sim = _simulate(c, state["seed"], geom)
        for name, dst in state["out"].items():
            sim.field_into(name, dst)
        i = geom.info()
        out = dict(state["out"], counts=np.array([i["n_fluid"], i["n_nodes"], i["n_links"]]), delta=i["delta"],
                   p=sim.info()["p"])
        sim.close()
        geom.close()
        return out
    if c["kind"] == "batch":
        sims = [s for _, s in state["boxes"]]
        lbm.step_batch(sims, c["steps"])
        eta = np.array([s.observables_noalloc()["eta"] for s in sims])
        for s, out in zip(sims, state["out"]):
            for name, dst in out.items():
                s.field_into(name, dst)
        return {"eta": eta, "boxes": state["out"]}
    sim = state["sim"]
    if c["kind"] == "poll":
        o = sim.observables(profiles=True, site_map=True)
        return {k: np.float64(o[k]) if k in SCALARS else o[k] for k in SCALARS + PROFILES + ("site_map",)}
    if c["kind"] == "step":
        sim.step(c["steps"])
    for name, dst in state["out"].items():
        sim.field_into(name, dst)
    return state["out"]


def work(case):
    """Every population read once and written once per step (the state and
    the outputs alone where there is no step); about ten operations per
    population."""
    c = dict(case)
    if c["kind"] == "batch":
        n = sum(s ** 3 for s in _sides(c))
        fluid = n * (0.5 + 0.5 * 0.65)  # (at the mean porosity)
    else:
        plane, n = c["nx"] * c["ny"], c["nx"] * c["ny"] * c["nz"]
        fluid = n - plane * (c["z1"] - c["z0"]) * (1 - c["porosity"])
        if c["sample"] == "plates":
            fluid = n - 2 * c["ny"] * (c["z1"] - c["z0"])
        elif c["sample"] == "disks":
            fluid = n - c["thickness"] * (c["z1"] - c["z0"]) * (1 - c["porosity"])
    pops = fluid * 19 * (1 + c["n_species"])
    size = 4 if c["storage"] == "fp32" else 2
    if c["kind"] == "batch":
        return {"bytes": c["steps"] * 2 * pops * size + 2 * 4 * n, "flops": c["steps"] * 10 * pops}
    if c["kind"] == "poll":
        return {"bytes": pops * size, "flops": 3 * pops}
    if c["kind"] == "snapshot":
        return {"bytes": pops * size + 4 * n * len(_names(c)), "flops": 3 * pops}
    if c["kind"] == "sample":
        # the mask, the initial populations and the two fields, written once;
        # 12 draws and 9 running sums per cell
        return {"bytes": n + pops * size + 2 * 4 * n, "flops": n * (12 * 8 + 9 * 2)}
    return {"bytes": c["steps"] * 2 * pops * size + 4 * n * len(_names(c)), "flops": c["steps"] * 10 * pops}


# ---- the same results in 64 bits, with plain torch -------------------------

CX = (0, 1, -1, 0, 0, 0, 0, 1, -1, 1, -1, 1, -1, 1, -1, 0, 0, 0, 0)
CY = (0, 0, 0, 1, -1, 0, 0, 1, -1, -1, 1, 0, 0, 0, 0, 1, -1, 1, -1)
CZ = (0, 0, 0, 0, 0, 1, -1, 0, 0, 0, 0, 1, -1, -1, 1, 1, -1, -1, 1)
W = (1 / 3,) + (1 / 18,) * 6 + (1 / 36,) * 12
OPP = (0,) + tuple(i + 1 if i & 1 else i - 1 for i in range(1, 19))
GAMMA = 0x9E3779B97F4A7C15


def _shift(a, i):
    """What lies at x - c_i, at x (every side taken as periodic: the open
    ends' planes are set apart)."""
    return torch.roll(a, (CZ[i], CY[i], CX[i]), (-3, -2, -1))


def _i64(v):
    return v - (1 << 64) if v >= 1 << 63 else v


def _splitmix(x):
    """SplitMix64's first output for state x (int64 tensors, wrapping)."""
    z = x + _i64(GAMMA)
    z = (z ^ ((z >> 30) & ((1 << 34) - 1))) * _i64(0xBF58476D1CE4E5B9)
    z = (z ^ ((z >> 27) & ((1 << 37) - 1))) * _i64(0x94D049BB133111EB)
    return z ^ ((z >> 31) & ((1 << 33) - 1))


def _chord(mask, z0, z1):
    """Mean pore chord length of the slab: 3 fluid cells / fluid runs along
    the axes, x and y periodic, z cut off at the slab."""
    f = mask[z0:z1] == 0
    n, runs = int(f.sum()), 0
    if n == 0:
        return 0.0
    for axis in (2, 1):
        runs += int((f & ~torch.roll(f, 1, axis)).sum()) + int(f.all(axis).sum())
    below = torch.cat([torch.zeros_like(f[:1]), f[:-1]])
    return 3.0 * n / (runs + int((f & ~below).sum()))


def _probability(c, mask):
    delta = _chord(mask, c["z0"], c["z1"])
    if c["p"] >= 0:
        return c["p"], delta
    return (min(1.0, math.sqrt(1 / 3) / (c["Da"] * delta)) if delta > 0 else 1.0), delta


def _generated(c, seed):
    """The synthetic sample: integer noise, nine running sums, the smallest
    values of the slab fluid."""
    nx, ny, nz, z0, z1 = c["nx"], c["ny"], c["nz"], c["z0"], c["z1"]
    cell = torch.arange(nx * ny * nz, device="cuda")
    v = torch.full_like(cell, -12 * 32768)
    for k in range(12):
        v += (_splitmix((cell * 12 + k) ^ seed) >> 48) & 0xFFFF
    v = v.reshape(nz, ny, nx)
    t = math.sqrt(2.0 * c["corr_len"] ** 2 + 1.0)
    width = min(range(1, int(t) + 4, 2), key=lambda w: (abs(t - w), w))
    for axis in (2, 1, 0):
        for _ in range(3):
            v = sum(torch.roll(v, d, axis) for d in range(-(width // 2), width // 2 + 1))
    slab = v[z0:z1].reshape(-1)
    m = torch.zeros((nz, ny, nx), dtype=torch.uint8, device="cuda")
    part = torch.ones_like(slab, dtype=torch.uint8)
    part[torch.sort(slab, stable=True)[1][:round(c["porosity"] * slab.numel())]] = 0
    m[z0:z1] = part.reshape(m[z0:z1].shape)
    return m


class _Exact:
    """Two-lattice statement of the method: collide, gather at the catalytic
    nodes, pull."""

    def __init__(self, c, seed, mask):
        self.c, self.mask = c, mask
        self.p, self.delta = _probability(c, mask)
        self.ns = 1 + c["n_species"]
        self.fluid = mask == 0
        self.node = mask == 1
        self.from_solid = [_shift(~self.fluid, i) for i in range(19)]
        self.from_node = [_shift(self.node, i) for i in range(19)]
        nz, ny, nx = mask.shape
        self.links = sum(_shift(self.fluid, j).to(torch.int8) for j in range(1, 19))
        self.f = torch.zeros((self.ns, 19, nz, ny, nx), dtype=torch.float64, device="cuda")
        for i in range(19):
            self.f[0, i] = W[i] * c["rho_out"]
            self.f[1, i] = W[i] * c["c_init"] * ~self.from_node[i]
        self.edge = torch.zeros((2, 3 + self.ns, ny, nx), dtype=torch.float64, device="cuda")
        self.hits = torch.zeros((2, nz, ny, nx), dtype=torch.float64, device="cuda")
        self.total = [0.0, 0.0]
        self.t = 0
        self.g = _force(c, seed)
        if c["random"]:
            key = _splitmix(torch.tensor(seed, device="cuda"))
            out = torch.stack([_shift(self.fluid, OPP[i]) for i in range(19)])  # x + c_i is fluid
            out[0] = False
            at = self.node & (self.links > 0)
            self.at, self.out, self.key = at, out[:, at], key
            self.cell = torch.arange(mask.numel(), device="cuda").reshape(mask.shape)[at]

    def moments(self):
        c = self.c
        rho = self.f.sum(1)
        j = []
        for e in (CX, CY, CZ):
            arrays = range(self.ns) if c["bary"] else (0,)
            j.append(sum(e[i] * self.f[a, i] for a in arrays for i in range(1, 19) if e[i]))
        over = rho.sum(0) if c["bary"] else rho[0]
        u = [x / over for x in j]
        u[2] = u[2] + 0.5 * self.g
        return rho, u

    def equilibrium(self, i, rho, u):
        cu = CX[i] * u[0] + CY[i] * u[1] + CZ[i] * u[2]
        return W[i] * rho * (1 + 3 * cu + 4.5 * cu * cu - 1.5 * (u[0] ** 2 + u[1] ** 2 + u[2] ** 2))

    def step(self):
        c, f = self.c, self.f
        rho, u = self.moments()
        om = [1 / c["tau"]] + [1 / (c["tau_s"] or c["tau"])] * 2
        edge = torch.stack([torch.cat([torch.stack([x[z] for x in u]), rho[:, z]]) for z in (1, -2)])
        ends = []
        for side, rho_c in ((0, c["rho_in"]), (1, c["rho_out"])):
            e = self.edge[side]
            v = [0.0 * e[0], 0.0 * e[0], 0.0 * e[0] + c["u_in"]] if side == 0 and c["u_in"] >= 0 else list(e[:3])
            dens = [torch.full_like(e[0], rho_c)] + [torch.full_like(e[0], c["c_in"] if a == 1 else 0.0) if side == 0 else e[3 + a]
                                                     for a in range(1, self.ns)]
            ends.append((v, dens))
        for i in range(19):
            for a in range(self.ns):
                x = f[a, i]
                x += om[a] * (self.equilibrium(i, rho[a], u) - x)
                if a == 0 and self.g:
                    cu = CX[i] * u[0] + CY[i] * u[1] + CZ[i] * u[2]
                    x += (1 - 0.5 * om[0]) * W[i] * (3 * (CZ[i] - u[2]) + 9 * cu * CZ[i]) * rho[0] * self.g
                for z, (v, dens) in ((0, ends[0]), (-1, ends[1])):
                    x[z] = self.equilibrium(i, dens[a], v)
                x.masked_fill_(~self.fluid, 0.0)
        # the catalytic nodes
        self.hits.zero_()
        for a in range(1, self.ns):
            for i in range(1, 19):
                self.hits[a - 1] += _shift(f[a, i], i)
            self.hits[a - 1] *= self.node
            self.total[a - 1] += float(self.hits[a - 1].sum())
        if c["random"]:
            rank = self.out.long().cumsum(0) - 1
            got = torch.zeros((2, 19, self.cell.numel()), dtype=torch.float64, device="cuda")
            b = self.out.long().sum(0)
            for j in range(1, 19):
                h = (_splitmix(((self.t << 40) + (self.cell << 5) + j) ^ self.key) >> 32) & 0xFFFFFFFF
                r = (h * b) >> 32
                to = (self.out & (rank == r)).to(torch.int8).argmax(0)
                for a in range(1, self.ns):
                    got[a - 1].scatter_add_(0, to[None], _shift(f[a, j], j)[self.at][None])
        # streaming; a pair of opposite directions at a time (bounce-back swaps them)
        pR = self.p * c["pS_R"]
        keep = (1 - pR if c["desorb"] else 1 - c["pS_R"], pR, 1 - c["pS_P"])
        for i in range(1, 19, 2):
            for a in range(self.ns):
                new = []
                for d in (i, i + 1):
                    x = torch.where(self.from_solid[d], f[a, OPP[d]], _shift(f[a, d], d))
                    if a:
                        if c["random"]:
                            R = torch.zeros_like(x)
                            R[self.at] = got[0, d]
                            if a == 2:
                                P = torch.zeros_like(x)
                                P[self.at] = got[1, d]
                        else:
                            b = self.links.clamp(min=1)
                            R, P = self.hits[0] / b, self.hits[1] / b if a == 2 else None
                        back = keep[0] * R if a == 1 else keep[1] * R + keep[2] * P
                        x = torch.where(self.from_node[d], _shift(back, d), x)
                    new.append(x)
                f[a, i], f[a, i + 1] = new
        self.edge = edge
        self.t += 1

    def fields(self, names):
        rho, u = self.moments()
        inside = self.fluid.clone()
        inside[0] = inside[-1] = False
        have = {"rho_C": rho[0], "drho_C": rho[0] - 1, "rho_R": rho[1], "ux": u[0], "uy": u[1], "uz": u[2]}
        if self.ns > 2:
            have["rho_P"] = rho[2]
        return {k: torch.where(inside, have[k], 0.0).reshape(-1) for k in names}

    def observables(self):
        c = self.c
        F = self.fields(["rho_C", "rho_R", "uz"] + ["rho_P"] * (self.ns > 2))
        shape = self.mask.shape
        z = {k: v.reshape(shape) for k, v in F.items()}
        P = z.get("rho_P", torch.zeros_like(z["rho_R"]))
        pR = self.p * c["pS_R"]
        out = {k: None for k in SCALARS}
        prof = {"rhoC_z": z["rho_C"], "rhoR_z": z["rho_R"], "rhoP_z": P, "phiP_z": P * z["uz"], "react_z": pR * self.hits[0]}
        prof = {k: v.sum((1, 2)) for k, v in prof.items()}
        out.update(prof, M_C=prof["rhoC_z"].sum(), M_R=prof["rhoR_z"].sum(), M_P=prof["rhoP_z"].sum(),
                   eta=prof["rhoP_z"][-2] / prof["rhoR_z"][1], hits_R=self.total[0], hits_P=self.total[1],
                   reacted=pR * self.total[0], stuck_R=0.0 if c["desorb"] else c["pS_R"] * (1 - self.p) * self.total[0],
                   delta=self.delta, p=self.p)
        out = {k: v if v is None else torch.as_tensor(v, dtype=torch.float64) for k, v in out.items()}
        out["site_map"] = pR * self.hits[0][self.node & (self.links > 0)]
        return out


def exact(case, seed):
    c = dict(case)
    if c["kind"] == "batch":
        if c["count"] * c["steps"] * c["side_hi"] ** 3 > 8e9:
            return None
        eta, boxes = [], []
        for m, s in _members(c, seed):
            e = _Exact(m, s, _mask(m, s))
            for _ in range(c["steps"]):
                e.step()
            boxes.append(e.fields(("rho_R", "rho_P")))
            eta.append(float(e.observables()["eta"]))
        return {"eta": np.array(eta), "boxes": boxes}
    cells = c["nx"] * c["ny"] * c["nz"]
    if c["kind"] == "sample":
        mask = _generated(c, _generator_seed(seed))
        p, delta = _probability(c, mask)
        fluid, node = mask == 0, mask == 1
        inside = fluid.clone()
        inside[0] = inside[-1] = False
        R = sum(W[i] * c["c_init"] * (~_shift(node, i)) for i in range(19))
        return {"rho_C": torch.where(inside, c["rho_out"], 0.0).double().reshape(-1),
                "rho_R": torch.where(inside, R, 0.0).double().reshape(-1), "counts": None, "delta": delta, "p": p}
    if cells > 8e7 or cells * c["steps"] > 1.6e9:
        return None
    if c["kind"] == "poll":
        c, seed = _polled(c, seed)
    e = _Exact(c, seed, _mask(c, seed))
    for _ in range(c["steps"]):
        e.step()
    return e.observables() if c["kind"] == "poll" else e.fields(_names(c))
