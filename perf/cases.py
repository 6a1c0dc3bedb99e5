"""What a user of the stepper has it do, as cases that can be timed.

A case is one job (or a short piece of one) through the public entry points:
the initial fields of a problem go in from device memory, the problem is
stepped, the final fields come back to device memory -- ``Sim.set_field``,
``Sim.step``, ``Sim.get_field``, and for several problems ``Batch``.  The
contexts (and their tuning) are made once, as a program that runs many jobs
keeps them.

Keys of a case:
  kind     "job" (one problem) or "batch" (several front problems stepped
           by shared launches)
  problem  a family of ``workloads``: diffusion, brusselator, turing, air,
           front, ch_table1, plume
  nx, ny, nz, steps, storage ("f32" / "bf16"), stencil (7 / 19)
  faces    "zero-flux" or "periodic" (Brusselator only; the other families
           have their own)
  kernel   "march" (the default) or "resident"
  tuned    the context is autotuned once after creation, as the benchmark
           does; otherwise the library's default tuning
  mass     the job ends with the conservation check (``Sim.mass``)
  members, lo, hi, edges_seed   a batch's cubes: edges drawn from lo..hi
"""
from __future__ import annotations

import math
import random

import torch

from paper_1004_0480_gb300 import workloads as W
from paper_1004_0480_gb300.sim import Batch, Sim

_SPECIES = {"diffusion": 1, "brusselator": 2, "turing": 2, "air": 3, "front": 3,
            "ch_table1": 3, "plume": 1}
# the plume starts here: its vertical wind sin(n dt / 500) is then at a
# general phase instead of zero
_PLUME_STEP0 = 250


def _job(name, problem, nx, ny, nz, steps, storage="f32", stencil=7, faces="zero-flux",
         kernel="march", tuned=False, mass=False):
    return dict(name=name, kind="job", problem=problem, nx=nx, ny=ny, nz=nz, steps=steps,
                storage=storage, stencil=stencil, faces=faces, kernel=kernel, tuned=tuned,
                mass=mass)


def listed():
    return [
        # a small problem watched closely: ten steps between two snapshots,
        # each with its conservation check (latency, launches)
        _job("watch-32", "diffusion", 32, 32, 32, 10, mass=True),
        # the 64^3 diffusion run of the benchmark on the kernel for grids
        # that stay in L2
        _job("diffusion-64-resident", "diffusion", 64, 64, 64, 100, kernel="resident"),
        # a small request as a program without any tuning makes it: sizes
        # that fit no tile, zero-flux walls
        _job("brusselator-odd", "brusselator", 97, 65, 50, 200),
        # the benchmark's headline problem, tuned as the benchmark tunes it
        _job("brusselator-256", "brusselator", 256, 256, 256, 100, faces="periodic", tuned=True),
        # the same with bfloat16 state
        _job("brusselator-256-bf16", "brusselator", 256, 256, 256, 100, storage="bf16",
             faces="periodic", tuned=True),
        # the paper's Turing system on its timing grid and its own stencil
        _job("turing-192-19pt", "turing", 192, 192, 192, 100, stencil=19),
        # the largest single field of the benchmark
        _job("diffusion-512", "diffusion", 512, 512, 512, 40, tuned=True),
        # atmospheric chemistry: wind, point source, different D per axis
        _job("air-512x512x64", "air", 512, 512, 64, 100, tuned=True),
        # one Cahn-Hilliard front at the largest edge of the batch workload
        _job("front-192", "front", 192, 192, 192, 60),
        # many uneven front problems stepped together
        dict(name="front-batch", kind="batch", problem="front", members=8, lo=48, hi=192,
             edges_seed=2, steps=60, storage="f32", stencil=7),
        # the paper's phase separation on its timing grid (two passes a step)
        _job("ch-table1-192-19pt", "ch_table1", 192, 192, 192, 60, stencil=19),
        # the paper's plume on its own grid: time-dependent 3-D wind
        _job("plume-144x144x384-19pt", "plume", 144, 144, 384, 100, stencil=19),
    ]


def draw(rng: random.Random):
    def edge(lo, hi):
        n = int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))
        return n if rng.random() < 0.5 else max(lo, n // 16 * 16)   # half of them round

    if rng.random() < 0.15:
        lo = edge(32, 96)
        return dict(kind="batch", problem="front", members=rng.randint(2, 10), lo=lo,
                    hi=rng.randint(lo, 192), edges_seed=rng.randrange(1 << 20),
                    steps=rng.randint(20, 80), storage=rng.choice(["f32", "f32", "bf16"]),
                    stencil=7)
    problem = rng.choice(["diffusion", "brusselator", "brusselator", "turing", "air", "front",
                          "ch_table1", "plume"])
    stencil = {"ch_table1": 19, "plume": rng.choice([7, 19]),
               "turing": rng.choice([7, 19, 19]), "brusselator": rng.choice([7, 7, 19])
               }.get(problem, 7)
    resident = stencil == 7 and problem in ("diffusion", "brusselator", "turing", "air") \
        and rng.random() < 0.15
    nx, ny, nz = (edge(16, 96) if resident else edge(24, 320) for _ in range(3))
    if problem == "air":
        nz = min(nz, 96)
    c = _job("", problem, nx, ny, nz, rng.randint(20, 120),
             storage="bf16" if rng.random() < 0.25 else "f32", stencil=stencil,
             faces=rng.choice(["zero-flux", "periodic"]) if problem == "brusselator"
             else "zero-flux",
             kernel="resident" if resident else "march",
             tuned=not resident and rng.random() < 0.3, mass=rng.random() < 0.2)
    # no more cell updates than the largest listed case
    cap = 512 ** 3 * 40
    c["steps"] = max(1, min(c["steps"], cap // (nx * ny * nz * _SPECIES[problem])))
    del c["name"]
    return c


# ------------------------------------------------------------------ problems
def _configs(case):
    """The problem of a job, or the problems of a batch's members."""
    p = case["problem"]
    if case["kind"] == "batch":
        edges = W.batch_sizes_ch(case["members"], case["lo"], case["hi"], case["edges_seed"])
        return [W.ch_front(n, steps=case["steps"]) for n in edges]
    shape = (case["nx"], case["ny"], case["nz"])
    if p == "diffusion":
        cfg = W.diffusion_blob(shape=shape)
    elif p == "brusselator":
        cfg = W.brusselator(shape=shape, bc="periodic" if case["faces"] == "periodic"
                            else "neumann")
    elif p == "turing":
        cfg = W.turing(shape=shape)
    elif p == "air":
        nx, ny, nz = shape
        cfg = W.air(shape, src=(nx // 8, ny // 2, min(2, nz - 1)))
    elif p == "front":
        cfg = W.ch_front(shape=shape)
    elif p == "ch_table1":
        cfg = W.ch_table1(shape=shape)
    elif p == "plume":
        cfg = W.plume(shape)
    else:
        raise ValueError(p)
    return [W.with_(cfg, stencil=case["stencil"], steps=case["steps"])]


def _inputs(problem, cfg, seed, member=0):
    """Fields (S, nz, ny, nx), float32 on the GPU, as the family meets them:
    its own start with seeded noise, or where that start is uniform (plume,
    ch_table1) a state from within a run."""
    nx, ny, nz = cfg["shape"]
    S = cfg["nspecies"]
    g = torch.Generator(device="cuda").manual_seed(1_000_003 * (int(seed) + 1) + member)
    u = torch.rand((S, nz, ny, nx), generator=g, device="cuda")
    z, y, x = (torch.arange(n, device="cuda", dtype=torch.float32) for n in (nz, ny, nx))
    z, y, x = z.view(nz, 1, 1), y.view(1, ny, 1), x.view(1, 1, nx)
    if problem == "diffusion":
        r2 = sum((a - (n - 1) / 2) ** 2 for a, n in ((x, nx), (y, ny), (z, nz)))
        u[0] += 10.0 * torch.exp(-r2 / 72.0)
    elif problem == "brusselator":
        a, b = cfg["params"]["a"], cfg["params"]["b"]
        for s, base in enumerate((a, b / a)):
            u[s] = base * (1.0 + 0.01 * (2.0 * u[s] - 1.0))
    elif problem == "turing":
        u = 1.0 + cfg["sigma"] * (2.0 * u - 1.0)
    elif problem == "air":
        for s, base in enumerate((0.01, 0.01, 1.0)):
            u[s] = base * (1.0 + 0.01 * (2.0 * u[s] - 1.0))
    elif problem == "front":
        u[0] = 0.0
        u[0, 0] = cfg["bc_value"][0][4]
        u[1] = 1.0
        u[2] = 0.005 * (2.0 * u[2] - 1.0)
    elif problem == "ch_table1":
        front = torch.exp(-x * (6.0 / nx))
        u[0] = 10.0 * front * (0.9 + 0.1 * u[0])
        u[0, :, :, 0] = cfg["bc_value"][0][0]
        u[1] = (1.0 - front) * (0.9 + 0.1 * u[1])
        u[2] = -1.0 + u[2]
    elif problem == "plume":
        src = cfg["source"]
        r2 = ((x - src["x"]) / 12) ** 2 + ((y - src["y"]) / 8) ** 2 + ((z - src["z"]) / 24) ** 2
        u[0] = 1000.0 * torch.exp(-0.5 * r2) * (0.95 + 0.1 * u[0])
    return u.contiguous()


def prepare(case, seed):
    cfgs = _configs(case)
    sims = [Sim(cfg, case["storage"]) for cfg in cfgs]
    state = dict(case=case, sims=sims, batch=None,
                 fields=[_inputs(case["problem"], cfg, seed, i) for i, cfg in enumerate(cfgs)])
    state["out"] = [torch.empty_like(f) for f in state["fields"]]
    if case["kind"] == "batch":
        state["batch"] = Batch("ch_front", case["storage"])
        for sim in sims:
            state["batch"].add(sim)
        return state
    sim = sims[0]
    if case["kernel"] != "march":
        sim.set_kernel(case["kernel"])
    if case["tuned"]:
        torch.cuda.synchronize()            # the fields were made on torch's stream
        sim.set_fields(state["fields"][0])
        sim.autotune()
    return state


def run(state):
    case = state["case"]
    for sim, f in zip(state["sims"], state["fields"]):
        sim.set_fields(f)
    sim = state["sims"][0]
    if state["batch"] is not None:
        state["batch"].step(case["steps"])
        state["batch"].sync()
    else:
        if case["problem"] == "plume":      # every job starts at the same time
            sim.lib.rd_set_step_count(sim.ctx, _PLUME_STEP0)
        sim.step(case["steps"])
    for m, o in zip(state["sims"], state["out"]):
        for s in range(m.nspecies):
            m.get_field(s, o[s])
    if case.get("mass"):
        return dict(fields=state["out"], mass=[list(sim.mass(s)) for s in range(sim.nspecies)])
    return dict(fields=state["out"])


# ---------------------------------------------------------------------- work
def _cells(case):
    if case["kind"] == "batch":
        edges = W.batch_sizes_ch(case["members"], case["lo"], case["hi"], case["edges_seed"])
        return sum(int(n) ** 3 for n in edges)
    return case["nx"] * case["ny"] * case["nz"]


def work(case):
    """Fields in and out once; floating-point operations of the scheme per
    cell and step (a fused multiply-add counts two)."""
    p, S, n = case["problem"], _SPECIES[case["problem"]], _cells(case)
    lap = 23 if case["stencil"] == 19 else 7          # sums and centre term
    aniso = 8 if p == "air" else 0                    # one D per axis
    react = {"diffusion": 0, "brusselator": 9, "turing": 10, "air": 5, "front": 2,
             "ch_table1": 6, "plume": 0}[p]
    wind = {"air": 3 * S, "plume": 9}.get(p, 0)
    # Cahn-Hilliard: the third species' transport is mu (Laplacian, its
    # polynomial and the sum) and the Laplacian of mu
    ch = lap + 6 if p in ("front", "ch_table1") else 0
    flops = S * (lap + aniso + 3) + react + wind + ch
    return {"bytes": 2 * 4 * S * n, "flops": flops * n * case["steps"]}


# --------------------------------------------------------------------- exact
def _shift(c, axis, d, periodic):
    """Neighbour values one cell along ``axis`` (d = -1 or +1); a zero-flux
    face repeats the face cell."""
    dim = 2 - axis                                    # fields are (z, y, x)
    if periodic:
        return torch.roll(c, -d, dim)
    n = c.shape[dim]
    if d < 0:
        return torch.cat([c.narrow(dim, 0, 1), c.narrow(dim, 0, n - 1)], dim)
    return torch.cat([c.narrow(dim, 1, n - 1), c.narrow(dim, n - 1, 1)], dim)


def _lap(c, cfg, per, D=None):
    """Laplacian of c; with D, sum_a D_a d2c/da2 (7-point)."""
    ih2 = 1.0 / (cfg["h"] * cfg["h"])
    if cfg.get("stencil", 7) == 19:
        t = -24.0 * c
        for a in range(3):
            for d in (-1, 1):
                f = _shift(c, a, d, per[a])
                t += 2.0 * f
                for b in range(a + 1, 3):
                    t += _shift(f, b, -1, per[b])
                    t += _shift(f, b, 1, per[b])
        return t * (ih2 / 6.0 * (D[0] if D else 1.0))
    t = torch.zeros_like(c)
    for a in range(3):
        w = ih2 * (D[a] if D else 1.0)
        t += w * (_shift(c, a, -1, per[a]) + _shift(c, a, 1, per[a]) - 2.0 * c)
    return t


def _upwind(c, axis, u, h, periodic):
    """-u dc/da, first order, from the side the wind comes from."""
    if u >= 0:
        return -u / h * (c - _shift(c, axis, -1, periodic))
    return -u / h * (_shift(c, axis, 1, periodic) - c)


def _rhs(cfg, f, per, n):
    S, h, q = cfg["nspecies"], cfg["h"], cfg["params"]
    kind = cfg["model"]
    r = [None] * S
    if kind == "diffusion":
        r = [torch.zeros_like(f[0])]
    elif kind == "brusselator":
        uuv = f[0] * f[0] * f[1]
        r = [q["a"] - (q["b"] + 1.0) * f[0] + uuv, q["b"] * f[0] - uuv]
    elif kind == "turing":
        r = [f[0] - f[0] ** 3 - f[1], q["gamma"] * (f[0] - q["alpha"] * f[1] - q["beta"])]
    elif kind == "air":
        net = q["j"] * f[1] - q["k"] * f[0] * f[2]
        r = [net, -net, net.clone()]
    elif kind == "ch_front":
        ab = q["k"] * f[0] * f[1]
        c = f[2]
        mu = 2.0 * c * (c - 1.0) * (2.0 * c - 1.0) - q["kappa"] * _lap(c, cfg, per)
        r = [-ab, -ab, ab + q["M"] * _lap(mu, cfg, per)]
    elif kind == "ch_table1":
        r1, r2 = q["k1"] * f[0] * f[1], q["k2"] * f[0] * f[2]
        c = f[2]
        inner = q["eps"] * c - q["gamma"] * c ** 3 + q["sigma"] * _lap(c, cfg, per)
        r = [-r1 - r2, -r1, r1 - r2 - q["lam"] * _lap(inner, cfg, per)]
    w, src = cfg["wind"], cfg["source"]
    for s in range(S):
        if any(cfg["D"][s]):
            r[s] = r[s] + _lap(f[s], cfg, per, cfg["D"][s])
        if w and w["kind"] == "log":
            nz = f[s].shape[0]
            uz = torch.log1p(torch.arange(nz, device=f[s].device, dtype=torch.float64))
            uz = (w["u0"] / math.log1p(nz) * uz).view(nz, 1, 1)
            r[s] = r[s] - uz / h * (f[s] - _shift(f[s], 0, -1, per[0]))
        elif w:
            vz = w["uz_amp"] * math.sin(n * cfg["dt"] / w["uz_tau"])
            for a, v in enumerate((w["ux"], w["uy"], vz)):
                r[s] = r[s] + _upwind(f[s], a, v, h, per[a])
        if src and src["species"] == s:
            r[s][src["z"], src["y"], src["x"]] += src["rate"]
    return r


def _hold(cfg, s, c):
    for face in (5, 4, 3, 2, 1, 0):
        if cfg["bc"][s][face] == "dirichlet":
            dim, last = 2 - face // 2, face & 1
            c.select(dim, c.shape[dim] - 1 if last else 0).fill_(cfg["bc_value"][s][face])


def _solve(cfg, fields, steps, n0):
    per = [cfg["bc"][0][2 * a] == "periodic" for a in range(3)]
    f = [x.double() for x in fields]
    for n in range(n0, n0 + steps):
        r = _rhs(cfg, f, per, n)
        f = [f[s] + cfg["dt"] * r[s] for s in range(cfg["nspecies"])]
        for s in range(cfg["nspecies"]):
            _hold(cfg, s, f[s])
    return torch.stack(f)


def exact(case, seed):
    out = []
    for i, cfg in enumerate(_configs(case)):
        x = _inputs(case["problem"], cfg, seed, i)
        out.append(_solve(cfg, x, case["steps"],
                          _PLUME_STEP0 if case["problem"] == "plume" else 0))
    if case.get("mass"):
        return dict(fields=out, mass=[[float(c.sum()), float(c.square().sum()), 0]
                                      for c in out[0]])
    return dict(fields=out)
