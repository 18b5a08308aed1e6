"""Workloads that time the library through its public entry points.

Each case is one call pattern of a user's program:

  kind "steps"   a simulation advanced by a host program: upload the state,
                 rebuild the lists, run `steps` time steps, read the state
                 and the forces back (one or more instances in a context)
  kind "sweep"   the same for a batch of equal-sized viscometers, with the
                 viscosity read-out of every instance after the steps, as the
                 surrogate's data generation does
  kind "stages"  one force evaluation by the stage calls (build, density, drag,
                 forces), as a program with its own integrator does
  kind "noalloc" the allocation-free density of one particle set
  kind "train"   one epoch of the surrogate network over `rows` samples
  kind "grad"    loss and gradients of one batch
  kind "infer"   predictions for `rows` query points

Lengths and physical constants are those of paper_2002_03120_gb300.cases and
surrogate (SI water or the mesoscale units); the positions are a lattice
disordered by 15 % of its spacing, about what a flow that has run for a while
looks like (the lattice's own 1 % holds for the first steps only), the
velocities a reverse-Poiseuille profile (or a falling column) plus a random
part.  Forces that were computed in FP32 (split precision), and the state
that carries their error after some steps, are handed on in FP32; the FP64
path's in FP64.
"""
import math

import numpy as np
import torch

from paper_2002_03120_gb300 import binding as B
from paper_2002_03120_gb300 import cases as C
from paper_2002_03120_gb300 import surrogate as S

FLUID, RIGID, INNER, OUTER = 0, 1, 2, 3


# ------------------------------------------------------------------ the cases
def listed():
    return [
        # the smallest full-size viscometer of the surrogate's data generation,
        # run on its own: 3,456 particles, launches and latency count
        {"name": "step_small_split", "kind": "steps", "shape": "flow", "prec": "split", "units": "meso",
         "nx": 12, "ny": 24, "inst": 1, "phi": 0.0, "mode": 0, "tpp": 4, "cells": 2, "steps": 10},
        # reverse Poiseuille 16x32x16 (8,192 particles), FP64, as created (no
        # tuning call): the plain first use of the library
        {"name": "poiseuille_fp64", "kind": "steps", "shape": "flow", "prec": "fp64", "units": "si",
         "nx": 16, "ny": 32, "inst": 1, "phi": 0.0, "mode": 1, "tpp": 1, "cells": 1, "steps": 5},
        # single-sphere sedimentation 32x32x64 between walls (73,728
        # particles), FP64 with the tuner's choice
        {"name": "sedimentation_fp64", "kind": "steps", "shape": "column", "prec": "fp64", "units": "si",
         "nx": 32, "nz": 64, "spheres": 1, "mode": 1, "tpp": 1, "cells": 2, "steps": 4},
        # dam break with spheres, friction, pressure filter and collision
        # viscosity in a walled tank (374,000 particles), split, tuned
        {"name": "dam_break_split", "kind": "steps", "shape": "dam", "prec": "split", "units": "si",
         "ny": 42, "spheres": 3000, "mode": 0, "tpp": 1, "cells": 2, "steps": 5},
        # 64 mesoscale viscometers of 12x24x12 in one context, 25 steps between
        # two read-outs: the surrogate's data generation
        {"name": "sweep_64_split", "kind": "sweep", "shape": "flow", "prec": "split", "units": "meso",
         "nx": 12, "ny": 24, "inst": 64, "phi": 0.3, "mode": 0, "tpp": 1, "cells": 2, "steps": 25},
        # uneven batched viscometers (fluid counts 20k-400k, solid fraction up
        # to 0.3, about 2M particles), split, tuned: the large production run
        {"name": "batch_12_split", "kind": "steps", "shape": "flow", "prec": "split", "units": "si",
         "nx": 58, "ny": 116, "inst": 12, "phi": 0.3, "mode": 0, "tpp": 1, "cells": 2, "steps": 5},
        # one force evaluation of a slurry instance by the stage calls, FP64, as created
        {"name": "stages_slurry_fp64", "kind": "stages", "shape": "flow", "prec": "fp64", "units": "si",
         "nx": 22, "ny": 44, "inst": 1, "phi": 0.2, "mode": 1, "tpp": 1, "cells": 1, "steps": 0},
        # the allocation-free density call on a mid-sized set
        {"name": "noalloc_46k", "kind": "noalloc", "nx": 29, "ny": 55},
        # one epoch of 2,000 samples at batch 256: seven full batches and a ragged one of 208
        {"name": "train_epoch_2000", "kind": "train", "rows": 2000, "batch": 256},
        # gradients at the largest batch the network takes
        {"name": "grad_4096", "kind": "grad", "rows": 4096, "batch": 4096},
        # proposal scoring: 10^6 query points
        {"name": "infer_1m", "kind": "infer", "rows": 1000000},
        # a re-check of a few proposals, odd size
        {"name": "infer_1001", "kind": "infer", "rows": 1001},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["flow", "flow", "flow", "column", "dam", "sweep", "stages", "stages", "noalloc", "train",
                       "grad", "infer"])
    split = rng.random() < 0.6
    base = {"prec": "split" if split else "fp64", "cells": rng.choice([1, 2]),
            "mode": rng.choice([0, 0, 1]) if split else 1, "tpp": 1}
    if kind in ("flow", "stages"):
        n = _log(rng, 12, 50 if split else 24)
        inst = rng.choice([1, 1, 2, 5]) if n < 30 else 1
        if n < 20 and base["mode"] == 0:
            base["tpp"] = rng.choice([1, 2, 4])
        return dict(base, kind="steps" if kind == "flow" else "stages", shape="flow",
                    units=rng.choice(["si", "meso"]), nx=n, ny=2 * n + rng.choice([-1, 0, 1]), inst=inst,
                    phi=round(rng.choice([0.0, rng.uniform(0.02, 0.3)]), 3), steps=rng.randint(1, 8) if kind == "flow" else 0)
    if kind == "column":
        return dict(base, kind="steps", shape="column", units="si", nx=_log(rng, 13, 32), nz=_log(rng, 20, 64),
                    spheres=rng.choice([1, 1, 7]), steps=rng.randint(1, 4))
    if kind == "dam":
        ny = _log(rng, 12, 42 if split else 20)
        return dict(base, kind="steps", shape="dam", units="si", ny=ny, spheres=max(1, ny ** 3 // 25),
                    steps=rng.randint(1, 5))
    if kind == "sweep":
        return dict(base, prec="split", mode=0, kind="sweep", shape="flow", units="meso", nx=12,
                    ny=24, inst=_log(rng, 4, 64), phi=0.3, steps=rng.randint(5, 25))
    if kind == "noalloc":
        return {"kind": "noalloc", "nx": _log(rng, 12, 38), "ny": rng.randint(24, 60)}
    if kind == "train":
        return {"kind": "train", "rows": rng.randint(100, 2000), "batch": rng.choice([64, 128, 256])}
    if kind == "grad":
        n = _log(rng, 32, 4096)
        return {"kind": "grad", "rows": n, "batch": n}
    return {"kind": "infer", "rows": _log(rng, 300, 900000)}


# ------------------------------------------------------------- particle sets
def _sub_lattice(nxyz, step, rng, count):
    """`count` distinct lattice sites (flat indices, x fastest) at least `step` apart on every axis."""
    ax = [np.arange(n // step) * step for n in nxyz]
    k, j, i = np.meshgrid(ax[2], ax[1], ax[0], indexing="ij")
    flat = ((k * nxyz[1] + j) * nxyz[0] + i).ravel()
    return rng.permutation(flat)[: min(count, len(flat))]


def _set(params, x, v, w, t, R, m):
    return dict(params=params, x=x, v=v, w=w, type=t, radius=R, mass=m)


def _spread(k):
    """0 for the first instance, then evenly spread in [0, 1): the sizes belong to the case, not to the seed."""
    return (k * 0.6180339887498949) % 1.0


def _flow(case, k, rng):
    """Reverse-Poiseuille box k of a case: n x ny x n fluid sites, spheres of
    diameter 3 dx replacing lattice sites up to the solid fraction."""
    nx, ny, inst = case["nx"], case["ny"], case["inst"]
    if inst > 1 and case["kind"] != "sweep":   # uneven sizes, log-uniform over a factor of 20 in particles
        f = 20.0 ** (-_spread(k) / 3.0)
        nx, ny = max(12, int(nx * f)), max(24, int(ny * f))
    phi = case["phi"] * (rng.uniform() if inst > 1 else 1.0)
    T = rng.uniform(280.0, 350.0)
    ratio = C.arrhenius_viscosity(T) / C.arrhenius_viscosity(293.15)
    if case["units"] == "meso":
        rho0, dx, eta = 3.0, 3.0 ** (-1.0 / 3.0), 25.0 * ratio
        p = C.base_params(dx=dx, rho0=rho0, eta=eta, alpha=7.0)
        p.update(p0=100.0, beta_p=100.0, kBT=0.01 * T / 293.15, r_c=3.9 * dx, lub_gap_min=0.1,
                 body_amp=10.0 ** rng.uniform(-1.0, 0.0))
        p["dt"] = S.meso_dt(p)
        vth, vflow = math.sqrt(p["kBT"]), 0.3
    else:
        dx = 1e-3
        p = C.base_params(dx=dx, eta=1e-3 * ratio)
        p.update(kBT=C.K_BOLTZMANN * T, body_amp=10.0 ** rng.uniform(-3.0, -1.0))
        vth, vflow = 1e-3, 1e-2
    p.update(box=[nx * dx, ny * dx, nx * dx], seed=int(rng.integers(1, 1 << 40)))
    x = C.lattice(nx, ny, nx, dx)
    n = len(x)
    x += rng.uniform(-0.15, 0.15, x.shape) * dx
    L = np.asarray(p["box"])
    x -= L * np.floor(x / L)
    x[x >= L] = 0.0
    v = rng.normal(0.0, vth, x.shape)
    s = 2.0 * x[:, 1] / L[1]
    v[:, 0] += vflow * np.where(s < 1.0, 4.0 * s * (1.0 - s), -4.0 * (s - 1.0) * (2.0 - s))
    w = rng.normal(0.0, 0.3 * vth / dx, x.shape)
    mf = p["rho0"] * dx ** 3
    t, R, m = np.zeros(n, np.int32), np.full(n, 0.5 * dx), np.full(n, mf)
    Rs = 1.5 * dx
    Vs = 4.0 / 3.0 * math.pi * Rs ** 3
    acc = _sub_lattice((nx, ny, nx), 3, rng, int(round(phi * n * dx ** 3 / Vs)))
    t[acc], R[acc], m[acc] = RIGID, Rs, 2.7 * p["rho0"] * Vs
    return _set(p, x, v, w, t, R, m)


def _with_walls(p, nxyz, sides, layers, parts, rng):
    dx = p["dx"]
    wx, wt = C._wall_layers(nxyz, dx, (0.0, 0.0, 0.0), layers, sides)
    nw, mf = len(wx), p["rho0"] * dx ** 3
    parts = parts + [(wx, np.zeros((nw, 3)), wt, np.full(nw, 0.5 * dx), np.full(nw, mf))]
    x, v, t, R, m = (np.concatenate([q[a] for q in parts]) for a in range(5))
    w = np.where((t <= RIGID)[:, None], rng.normal(0.0, 0.3, x.shape), 0.0)
    return _set(p, x, v, w, t.astype(np.int32), R, m)


def _fluid_and_spheres(p, nxyz, count, Rs_of, rho_s, v0, rng, periodic):
    """A disordered lattice block at the origin with spheres on some of its sites."""
    dx = p["dx"]
    x = C.lattice(*nxyz, dx)
    n = len(x)
    step = int(math.ceil(2.0 * Rs_of(64).max() / dx))
    acc = _sub_lattice(nxyz, step, rng, count) if count > 1 else np.array(
        [((nxyz[2] * 3 // 4) * nxyz[1] + nxyz[1] // 2) * nxyz[0] + nxyz[0] // 2])
    x += rng.uniform(-0.15, 0.15, x.shape) * dx
    for a in range(3):
        if periodic[a]:
            L = p["box"][a]
            x[:, a] -= L * np.floor(x[:, a] / L)
    v = rng.normal(0.0, 2e-3, x.shape) + np.asarray(v0)
    t, R, m = np.zeros(n, np.int32), np.full(n, 0.5 * dx), np.full(n, p["rho0"] * dx ** 3)
    Rs = Rs_of(len(acc))
    t[acc], R[acc], m[acc] = RIGID, Rs, rho_s * 4.0 / 3.0 * math.pi * Rs ** 3
    return (x, v, t, R, m)


def _column(case, rng):
    nx, nz, dx = case["nx"], case["nz"], 1e-3
    p = C.base_params(dx=dx)
    p.update(box=[nx * dx, nx * dx, nz * dx], periodic=[1, 1, 0], g=[0.0, 0.0, -9.81], artvis=1, dem_law=1,
             kn=1e3, restitution=0.9, seed=int(rng.integers(1, 1 << 40)))
    part = _fluid_and_spheres(p, (nx, nx, nz), case["spheres"], lambda k: np.full(k, 2.0 * dx), 2500.0,
                              (0.0, 0.0, 0.0), rng, p["periodic"])
    return _with_walls(p, (nx, nx, nz), [(2, 0), (2, 1)], 4, [part], rng)


def _dam(case, rng):
    ny = case["ny"]
    dx = 0.2 / 63
    p = C.base_params(dx=dx, dt=2e-5, c_sound=20.0)
    nxt, nzt = 5 * ny, 3 * ny
    p.update(box=[nxt * dx, ny * dx, nzt * dx], periodic=[0, 0, 0], g=[0.0, 0.0, -9.81], artvis=1,
             pressure_filter=1, clamp_negative_p=1, dem_law=1, kn=1e3, restitution=0.9, mu_fric=0.3,
             seed=int(rng.integers(1, 1 << 40)))
    part = _fluid_and_spheres(p, (2 * ny, ny, ny), case["spheres"],
                              lambda k: rng.uniform(1.5e-3, 2.5e-3, k), 2600.0, (0.3, 0.0, -0.1), rng,
                              p["periodic"])
    return _with_walls(p, (nxt, ny, nzt), [(0, 0), (0, 1), (1, 0), (1, 1), (2, 0)], 3, [part], rng)


def _instances(case, seed):
    rng = np.random.default_rng(seed)
    if case["shape"] == "flow":
        return [_flow(case, k, rng) for k in range(case["inst"])]
    return [_column(case, rng) if case["shape"] == "column" else _dam(case, rng)]


# --------------------------------------------------------------- the programs
def _net_data(case, seed):
    g = torch.Generator(device="cuda").manual_seed(seed)
    X = torch.rand((case["rows"], 3), generator=g, device="cuda")
    # log viscosity against solid fraction, temperature and forcing, with scatter
    T = 2.0 * X[:, 0] - 1.2 * X[:, 1] + 0.2 * torch.sin(3.0 * X[:, 2]) + 0.05 * torch.randn(
        case["rows"], generator=g, device="cuda")
    return X, T


def _noalloc_inputs(case, seed):
    rng = np.random.default_rng(seed)
    c = _flow(dict(nx=case["nx"], ny=case["ny"], inst=1, kind="noalloc", phi=0.0, units="si"), 0, rng)
    return c["params"], c["x"], c["type"]


def prepare(case, seed):
    kind = case["kind"]
    if kind in ("steps", "sweep", "stages"):
        insts = _instances(case, seed)
        split = case["prec"] == "split"
        sim = B.Sim(insts, precision=B.SDPD_PREC_SPLIT if split else B.SDPD_PREC_FP64)
        if case["mode"] != 1:
            sim.set_force_mode(case["mode"])
        if case["tpp"] != 1:
            sim.set_threads_per_particle(case["tpp"])
        if case["cells"] != 1:
            sim.set_cell_factor(case["cells"])
        x, v, w = (torch.tensor(np.concatenate([c[a] for c in insts]), device="cuda") for a in ("x", "v", "w"))
        out = [torch.empty((sim.N, 3), dtype=torch.float64, device="cuda") for _ in range(5)]
        return dict(case=case, sim=sim, x=x, v=v, w=w, out=out, split=split)
    if kind == "noalloc":
        p, x, t = _noalloc_inputs(case, seed)
        n = len(x)
        return dict(case=case, params=p, x=torch.tensor(x, device="cuda"), t=torch.tensor(t, device="cuda"),
                    d=torch.empty(n, dtype=torch.float64, device="cuda"),
                    p=torch.empty(n, dtype=torch.float64, device="cuda"))
    X, T = _net_data(case, seed)
    net = B.Mlp(seed=seed, batch_max=case.get("batch", 256))
    return dict(case=case, net=net, X=X, T=T, Y=torch.empty(case["rows"], device="cuda"))


def run(s):
    case = s["case"]
    kind = case["kind"]
    if kind in ("steps", "sweep", "stages"):
        sim = s["sim"]
        x, v, w, F, N = s["out"]
        sim.upload_state(s["x"], s["v"], s["w"])
        if kind == "stages":
            sim.evaluate(1)
            sim.download_state(F=F, N=N)
            return {"F": F.float(), "N": N.float()} if s["split"] else {"F": F, "N": N}
        sim.build_cells()
        sim.step(case["steps"])
        mu = [sim.viscosity_probe(k, 24)[1] for k in range(sim.n_inst)] if kind == "sweep" else []
        sim.download_state(x, v, w, F, N)
        out = {n: a.float() if s["split"] else a for n, a in zip("xvwFN", (x, v, w, F, N))}
        if mu:
            out["mu"] = np.asarray(mu, dtype=np.float32)
        return out
    if kind == "noalloc":
        B.density_noalloc(s["params"], s["x"], s["t"], s["d"], s["p"])
        return {"d": s["d"], "p": s["p"]}
    net, X, T = s["net"], s["X"], s["T"]
    if kind == "infer":
        net.infer(X, s["Y"])
        return s["Y"]
    if kind == "grad":
        loss = net.gradients(X, T)
        return {"loss": np.float32(loss), "g": net.grads()}
    b = case["batch"]
    for i in range(0, case["rows"], b):
        net.train_step(X[i:i + b], T[i:i + b], lr=1e-3, want_loss=False)
    return net.params()


# ------------------------------------------------------------------ the floor
NET = S.flops_per_query()
PAIRS = 0.5 * 4.0 / 3.0 * math.pi * 3.9 ** 3   # unordered pairs a particle at one particle per dx^3


def _mobile_and_all(case):
    """Mobile particles and all particles of a case."""
    if case["shape"] == "flow":
        n = case["nx"] ** 2 * case["ny"]
        if case["inst"] > 1 and case["kind"] != "sweep":
            n *= sum(20.0 ** -_spread(k) for k in range(case["inst"]))
        else:
            n *= case["inst"]
        return int(n), int(n)
    if case["shape"] == "column":
        n = case["nx"] ** 2 * case["nz"]
        return n, n + 8 * case["nx"] ** 2
    ny = case["ny"]
    return 2 * ny ** 3, 2 * ny ** 3 + (5 * ny + 6) * (ny + 6) * (3 * ny + 3) - 15 * ny ** 3


def work(case):
    kind = case["kind"]
    if kind in ("steps", "sweep", "stages"):
        mob, n = _mobile_and_all(case)
        evals = 1 if kind == "stages" else 2 * case["steps"]
        out = 2 if kind == "stages" else 5
        # 160 operations a pair and force evaluation (the pair forces with their
        # six normals), 20 a pair and density; x, v, w in, the results out
        return {"bytes": float((3 + out) * 24 * n), "flops": float(mob * PAIRS * 180 * evals)}
    if kind == "noalloc":
        n = case["nx"] ** 2 * case["ny"]
        return {"bytes": float(n * (24 + 4 + 16)), "flops": float(n * 2 * PAIRS * 20)}
    if kind == "infer":
        return {"bytes": float(16 * case["rows"]), "flops": float(NET * case["rows"])}
    par = 50177
    if kind == "grad":
        return {"bytes": float(16 * case["rows"] + 8 * par), "flops": float(3 * NET * case["rows"])}
    steps = -(-case["rows"] // case["batch"])
    return {"bytes": float(16 * case["rows"] + 24 * par * steps), "flops": float(3 * NET * case["rows"])}


# ------------------------------------------------- the same in 64 bits by torch
def exact(case, seed):
    kind = case["kind"]
    if kind == "noalloc":
        p, x, t = _noalloc_inputs(case, seed)
        if len(x) > 60000:
            return None
        d = _density(p, torch.tensor(x, device="cuda"), None)
        return {"d": d, "p": _pressure(p, d)}
    if kind in ("infer", "grad", "train"):
        return _exact_net(case, seed)
    if case["shape"] != "flow" or case["phi"] > 0.0 or case["inst"] > 1 or case["nx"] ** 2 * case["ny"] > 40000:
        return None
    c = _instances(case, seed)[0]
    p = c["params"]
    x, v, w = (torch.tensor(c[a], device="cuda") for a in ("x", "v", "w"))
    m = p["rho0"] * p["dx"] ** 3
    inertia = 0.4 * m * (0.5 * p["dx"]) ** 2
    L = torch.tensor(p["box"], dtype=torch.float64, device="cuda")
    if kind == "stages":
        F, N = _forces(p, x, v, w, 0)
        return {"F": F, "N": N}
    h = 0.5 * p["dt"]
    for n in range(case["steps"]):
        for half in (1, 2):
            F, N = _forces(p, x, v, w, n)
            v, w = v + h * F / m, w + h * N / inertia
            if half == 1:
                x = x + p["dt"] * v
                x = x - L * torch.floor(x / L)
    out = {"x": x, "v": v, "w": w, "F": F, "N": N}
    if kind == "sweep":
        out["mu"] = None
    return out


def _lucy_norm(p):
    h, dx = p["r_c"], p["dx"]
    n = int(math.ceil(h / dx)) + 1
    a = torch.arange(-n, n + 1, dtype=torch.float64)
    r = (a[:, None, None] ** 2 + a[None, :, None] ** 2 + a[None, None, :] ** 2).sqrt() * dx
    return 1.0 / (dx ** 3 * float(_lucy(r[r < h], h).sum()))


def _lucy(r, h):
    q = r / h
    return 105.0 / (16.0 * math.pi * h ** 3) * (1.0 + 3.0 * q) * (1.0 - q) ** 3


def _all_pairs(p, x):
    """Ordered pairs (i, j) within h of a periodic box and r_i - r_j, by chunks of brute force."""
    L = torch.tensor(p["box"], dtype=torch.float64, device=x.device)
    for i0 in range(0, len(x), 512):
        d = x[i0:i0 + 512, None, :] - x[None, :, :]
        d = d - L * torch.round(d / L)
        r2 = (d * d).sum(-1)
        i, j = torch.nonzero(r2 < p["r_c"] ** 2, as_tuple=True)
        off = i + i0 != j
        i, j = i[off], j[off]
        yield i + i0, j, d[i, j]


def _density(p, x, pairs):
    d = torch.full((len(x),), float(_lucy(torch.zeros(1, dtype=torch.float64), p["r_c"])), dtype=torch.float64, device=x.device)
    for i, j, r in (_all_pairs(p, x) if pairs is None else pairs):
        d.index_add_(0, i, _lucy(r.norm(dim=1), p["r_c"]))
    return _lucy_norm(p) * d


def _pressure(p, d):
    return p["p0"] * (d * p["dx"] ** 3) ** p["alpha"] - p["beta_p"]


def _philox(lo, hi, step, block, k0, k1):
    """Philox4x32-10 of the counters (lo, hi, step, block), words as int64 tensors."""
    M = 0xFFFFFFFF
    c = [lo, hi, torch.full_like(lo, step), torch.full_like(lo, block)]

    def mul(a, b):   # 32 x 32 -> (high, low), in halves that int64 holds
        al, ah = a & 0xFFFF, a >> 16
        t = al * b
        u = ah * b + (t >> 16)
        return (u >> 16) & M, ((u & 0xFFFF) << 16) | (t & 0xFFFF)

    for _ in range(10):
        h0, l0 = mul(c[0], 0xD2511F53)
        h1, l1 = mul(c[2], 0xCD9E8D57)
        c = [h1 ^ c[1] ^ k0, l1, h0 ^ c[3] ^ k1, l0]
        k0, k1 = (k0 + 0x9E3779B9) & M, (k1 + 0xBB67AE85) & M
    return c


def _normals(i, j, p, step):
    lo, hi = torch.minimum(i, j), torch.maximum(i, j)
    k0, k1 = p["seed"] & 0xFFFFFFFF, (p["seed"] >> 32) & 0xFFFFFFFF
    u = [((b >> 9).double() + 0.5) / 8388608.0 for q in (0, 1) for b in _philox(lo, hi, step, q, k0, k1)]
    z = []
    for a in (0, 2, 4):
        r, t = (-2.0 * u[a].log()).sqrt(), 2.0 * math.pi * u[a + 1]
        z += [r * t.cos(), r * t.sin()]
    return z


def _forces(p, x, v, w, step):
    """Force and torque of every particle of a fluid-only periodic box (pair
    forces C, D, R and T, the body force)."""
    pairs = list(_all_pairs(p, x))
    d = _density(p, x, pairs)
    pr = _pressure(p, d)
    h, eta, xi, kBT = p["r_c"], p["eta"], p["xi"], p["kBT"]
    Ca, Cb = 20.0 * eta / 3.0 - 4.0 * xi, 17.0 * xi - 40.0 * eta / 3.0
    F, N = torch.zeros_like(x), torch.zeros_like(x)
    for i, j, rv in pairs:
        r = rv.norm(dim=1, keepdim=True)
        e = rv / r
        Fk = 315.0 / (4.0 * math.pi * h ** 5) * (1.0 - r / h) ** 2
        di, dj = d[i, None], d[j, None]
        ga, gb = Ca * Fk / (di * dj), Cb * Fk / (di * dj)
        vij = v[i] - v[j]
        ev = (e * vij).sum(1, keepdim=True)
        f = p["coeff_c"] * (pr[i, None] / di ** 2 + pr[j, None] / dj ** 2) * Fk * rv
        f = f - p["coeff_d"] * (ga * (vij + e * ev / 3.0) + 2.0 / 3.0 * gb * e * ev)
        f = f - p["coeff_r"] * 0.5 * ga * torch.cross(rv, w[i] + w[j], dim=1)
        z = _normals(i, j, p, step)
        q = math.sqrt(0.5)
        W = torch.stack([torch.stack([z[0], q * z[3], q * z[4]], -1), torch.stack([q * z[3], z[1], q * z[5]], -1),
                         torch.stack([q * z[4], q * z[5], z[2]], -1)], 1)
        tr = (z[0] + z[1] + z[2])[:, None] / 3.0
        We = (W * e[:, None, :]).sum(-1)
        sa, sb = 2.0 * (kBT * ga).sqrt(), 2.0 * (kBT * gb.clamp_min(0.0)).sqrt()
        f = f + p["coeff_t"] / math.sqrt(p["dt"]) * (sa * (We - tr * e) + sb * tr * e)
        F.index_add_(0, i, f)
        N.index_add_(0, i, torch.cross(-0.5 * p["dx"] * e, f, dim=1))
    m, a = p["rho0"] * p["dx"] ** 3, p["split_axis"]
    F[:, p["body_axis"]] += m * torch.where(x[:, a] < 0.5 * p["box"][a], p["body_amp"], -p["body_amp"])
    return F, N


def _exact_net(case, seed):
    """The network in 64 bits throughout (no BF16 operands), with Adam as published."""
    X, T = (a.double() for a in _net_data(case, seed))
    net = B.Mlp(seed=seed, batch_max=256)
    P = torch.tensor(net.params(), dtype=torch.float64, device="cuda")   # the initial weights: an input
    net.close()

    def forward(P, X):
        o, y = 0, X
        for k, (a, b) in enumerate([(3, 128), (128, 128), (128, 128), (128, 128), (128, 1)]):
            y = y @ P[o:o + a * b].view(b, a).T + P[o + a * b:o + a * b + b]
            o += a * b + b
            if k < 4:
                y = torch.nn.functional.gelu(y)
        return y[:, 0]

    if case["kind"] == "infer":
        return torch.cat([forward(P, X[i:i + 100000]) for i in range(0, len(X), 100000)])
    m, q, t = torch.zeros_like(P), torch.zeros_like(P), 0
    b = case["batch"]
    for i in range(0, len(X), b):
        Q = P.clone().requires_grad_(True)
        loss = ((forward(Q, X[i:i + b]) - T[i:i + b]) ** 2).mean()
        g, = torch.autograd.grad(loss, Q)
        if case["kind"] == "grad":
            return {"loss": float(loss.detach()), "g": g}
        t += 1
        m, q = 0.9 * m + 0.1 * g, 0.999 * q + 0.001 * g * g
        P = P - 1e-3 * (m / (1 - 0.9 ** t)) / ((q / (1 - 0.999 ** t)).sqrt() + 1e-8)
    return P
