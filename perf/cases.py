"""Performance cases of the hybrid Shakhov / DSMC particle step.

What a user's program has the library do, through the Python binding: advance
a flow by a number of steps and read its fields (per step, every few steps,
or time-averaged), restart a flow from host particles, and sort cell keys
that the program owns.  Flows are those of
``paper_2506_23917_gb300.workloads``.

A program that advances a large flow tunes the collision schedule once and
keeps it (``tune``): here on a context of its own, so that the trial steps do
not move the measured flow.
"""
from __future__ import annotations

import math

import numpy as np
import torch

import paper_2506_23917_gb300 as sp
from paper_2506_23917_gb300 import workloads as W

PREC = {"fp64": sp.FP64, "fp32": sp.FP32, "fp32c": sp.FP32_CELL32}
NF = len(sp.FIELDS)
_cfg = {}       # meshes and cut-cell volumes, which do not depend on the seed
_schedule = {}  # tuned collision schedules


def listed():
    return [
        # a space-homogeneous relaxation of 1000 particles, read after every
        # step as a coupled program does: the smallest call there is
        {"name": "relax_fp64_1k", "kind": "relax", "n": 1000, "kn": 1e-2, "precision": "fp64", "steps": 1,
         "develop": 5, "tune": False, "read": "now", "mode": 0, "subcells": 0, "ntc_carry": 0},
        # the Sod tube of the parity configuration (200 cells, 100 / 12.5
        # particles per cell, FP64, 400 steps), 20 steps between two reads
        {"name": "sod_fp64_11k", "kind": "sod", "cells": 200, "ppc": 100.0, "kn": 1e-3, "precision": "fp64",
         "steps": 20, "develop": 20, "tune": False, "read": "now", "mode": 0, "subcells": 0, "ntc_carry": 0},
        # the headline flow: hypersonic cylinder, 600 x 300 cells, 40 per
        # cell, FP32 state, averaging while it runs
        {"name": "cylinder_fp32", "kind": "cylinder", "scale": 1.0, "ppc": 40.0, "kn": 0.01, "precision": "fp32",
         "steps": 20, "develop": 600, "tune": True, "read": "mean", "mode": 0, "subcells": 0, "ntc_carry": 0},
        # the same flow in FP64 (the precision that matches the oracle)
        {"name": "cylinder_fp64", "kind": "cylinder", "scale": 0.5, "ppc": 40.0, "kn": 0.01, "precision": "fp64",
         "steps": 5, "develop": 200, "tune": True, "read": "now", "mode": 0, "subcells": 0, "ntc_carry": 0},
        # the opt-in FP32 per-cell arithmetic
        {"name": "cylinder_cell32", "kind": "cylinder", "scale": 0.7, "ppc": 40.0, "kn": 0.01,
         "precision": "fp32c", "steps": 20, "develop": 400, "tune": True, "read": "now", "mode": 0, "subcells": 0,
         "ntc_carry": 0},
        # sonic jet into vacuum: occupancy from 0 to about 1500 per cell
        {"name": "jet_fp32", "kind": "jet", "scale": 0.5, "ppc": 1500.0, "kn": 0.02, "precision": "fp32",
         "steps": 10, "develop": 600, "tune": True, "read": "mean", "mode": 0, "subcells": 0, "ntc_carry": 0},
        # 3-D sphere with cut cells, about 30 million particles
        {"name": "sphere_fp32", "kind": "sphere", "scale": 0.625, "ppc": 30.0, "kn": 0.005, "precision": "fp32",
         "steps": 10, "develop": 100, "tune": True, "read": "now", "mode": 0, "subcells": 0, "ntc_carry": 0},
        # body-fitted cylinder mesh: point location by face crossing
        {"name": "ogrid_fp32", "kind": "ogrid", "nr": 150, "nt": 600, "ppc": 40.0, "kn": 0.05,
         "precision": "fp32", "steps": 10, "develop": 300, "tune": True, "read": "mean", "mode": 0, "subcells": 0,
         "ntc_carry": 0},
        # an ensemble of 64 independent tubes and boxes of uneven size in one
        # context, the averaged fields of every instance read at the end
        {"name": "ensemble_fp32", "kind": "ensemble", "instances": 64, "nmin": 1000, "nmax": 500000,
         "precision": "fp32", "steps": 50, "develop": 20, "tune": True, "read": "mean", "mode": 0, "subcells": 0,
         "ntc_carry": 0},
        # the whole call from host memory: state from page-locked memory, one
        # step, fields back to page-locked memory
        {"name": "cylinder_upload_step", "kind": "restart", "scale": 0.7, "ppc": 40.0, "kn": 0.01,
         "precision": "fp32", "steps": 1, "develop": 300, "tune": True, "read": "now", "mode": 0, "subcells": 0,
         "ntc_carry": 0},
        # an FP64 state in arbitrary order uploaded, indexed and reduced to
        # its moments
        {"name": "sphere_upload_fp64", "kind": "upload", "scale": 0.25, "ppc": 30.0, "kn": 0.005},
        # cell keys of a moved 2-D state, sorted in the caller's buffers
        {"name": "sort_16m", "kind": "sort", "nx": 512, "ny": 512, "keys": 16000000},
    ]


def _log(rng, a, b):
    return math.exp(rng.uniform(math.log(a), math.log(b)))


def draw(rng):
    kind = rng.choice(["relax", "sod", "cylinder", "cylinder", "jet", "sphere", "ogrid", "ensemble", "restart",
                       "upload", "sort"])
    if kind == "sort":
        return {"kind": kind, "nx": int(_log(rng, 20, 700)), "ny": int(_log(rng, 20, 700)),
                "keys": int(_log(rng, 2e4, 1.6e7))}
    if kind == "upload":
        return {"kind": kind, "scale": round(rng.uniform(0.06, 0.25), 4), "ppc": round(rng.uniform(8.0, 30.0), 2),
                "kn": 0.005}
    c = {"kind": kind, "precision": rng.choice(["fp32", "fp32", "fp32c", "fp64"]), "read": rng.choice(["now", "mean"]),
         "mode": rng.choice([0, 0, 0, 1, 2]), "subcells": rng.choice([0, 0, 0, 2]), "ntc_carry": rng.choice([0, 0, 1])}
    dbl = c["precision"] == "fp64"
    if kind == "relax":
        c.update(n=int(_log(rng, 500, 200000)), kn=_log(rng, 1e-4, 1.0), steps=rng.randint(1, 10), develop=5,
                 tune=False)
    elif kind == "sod":
        c.update(cells=int(_log(rng, 50, 5000)), ppc=round(_log(rng, 20.0, 500.0), 2), kn=_log(rng, 1e-4, 1e-1),
                 steps=rng.randint(5, 20), develop=20, tune=rng.choice([False, True]))
    elif kind in ("cylinder", "restart"):
        c.update(scale=round(_log(rng, 0.08, 0.5 if dbl else 0.9), 4), ppc=round(rng.uniform(15.0, 42.0), 2),
                 kn=_log(rng, 5e-3, 1e-1), steps=1 if kind == "restart" else rng.randint(2, 5 if dbl else 20),
                 develop=100, tune=rng.choice([False, True]))
        if kind == "restart":
            c["scale"] = min(c["scale"], 0.7)
    elif kind == "jet":
        c.update(scale=round(_log(rng, 0.1, 0.3 if dbl else 0.5), 4), ppc=round(_log(rng, 50.0, 1500.0), 2), kn=0.02,
                 steps=rng.randint(2, 4 if dbl else 10), develop=100, tune=rng.choice([False, True]))
    elif kind == "sphere":
        c.update(scale=round(rng.uniform(0.1, 0.25 if dbl else 0.5), 4), ppc=round(rng.uniform(10.0, 30.0), 2),
                 kn=0.005, steps=rng.randint(2, 4 if dbl else 10), develop=60, tune=rng.choice([False, True]))
    elif kind == "ogrid":
        c.update(nr=rng.randint(30, 80 if dbl else 150), nt=rng.randint(60, 200 if dbl else 600),
                 ppc=round(rng.uniform(15.0, 40.0), 2), kn=0.05, steps=rng.randint(2, 5 if dbl else 10), develop=60,
                 tune=rng.choice([False, True]), subcells=0)
    else:
        c.update(instances=rng.randint(8, 60), nmin=1000, nmax=100000 if dbl else 500000,
                 steps=rng.randint(2, 5 if dbl else 40), develop=10, tune=rng.choice([False, True]))
    return c


def _sizes(case):
    """Particle counts and Knudsen numbers of an ensemble: the case's, whatever the seed."""
    g = np.random.Generator(np.random.PCG64(1))
    n = case["instances"]
    return (np.exp(g.uniform(math.log(case["nmin"]), math.log(case["nmax"]), n)).astype(int),
            np.exp(g.uniform(math.log(1e-4), math.log(1.0), n)))


def _flow(case):
    """(config, regions) of a flow, built once per case."""
    key = tuple(sorted((k, v) for k, v in case.items() if k not in ("name", "steps", "develop", "tune", "read")))
    if key not in _cfg:
        k = case["kind"]
        if k == "sod":
            f = W.sod(ncell=case["cells"], ppc_left=case["ppc"], lam_left=case["kn"], n_steady=0)
        elif k in ("cylinder", "restart"):
            f = W.cylinder(scale=case["scale"], ppc=case["ppc"], Kn=case["kn"], n_steady=0)
        elif k == "jet":
            f = W.jet(scale=case["scale"], ppc=case["ppc"], Kn=case["kn"], plenum=1.0, n_steady=0)
        elif k in ("sphere", "upload"):
            f = W.sphere(scale=case["scale"], ppc=case["ppc"], Kn=case["kn"], n_steady=0)
        else:
            f = W.cylinder_ogrid(nr=case["nr"], nt=case["nt"], ppc=case["ppc"], Kn=case["kn"], n_steady=0,
                                 growth=1.005)
        if len(_cfg) > 16:
            _cfg.clear()
        _cfg[key] = f
    return _cfg[key]


def _particles(cfg, regions, seed, dtype):
    """Uniform positions outside the body, drifting Maxwellian velocities; page-locked host tensors."""
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    dim, P, V = cfg["dim"], [], []
    for r in regions:
        lo = list(r["lo"]) + [cfg["lo"][d] for d in range(len(r["lo"]), 3)]
        hi = list(r["hi"]) + [cfg["hi"][d] for d in range(len(r["hi"]), 3)]
        m = int(round(r["n"] * math.prod(hi[d] - lo[d] for d in range(3)) / cfg["Fn"]))
        x = torch.rand((dim, m), generator=g, device="cuda", dtype=torch.float64)
        for d in range(dim):
            x[d] = lo[d] + (hi[d] - lo[d]) * x[d]
        if cfg["body"] != W.BODY_NONE:
            r2 = sum((x[a] - cfg["body_c"][a]) ** 2 for a in range(2 if cfg["body"] == W.BODY_CIRCLE else 3))
            x = x[:, r2 >= cfg["body_r"] ** 2]
        v = torch.randn((3, x.shape[1]), generator=g, device="cuda", dtype=torch.float64)
        v = v * math.sqrt(cfg["R"] * r["T"]) + torch.tensor(r["u"], device="cuda", dtype=torch.float64)[:, None]
        P.append(x.to(dtype))
        V.append(v.to(dtype))
    return torch.cat(P, 1).cpu().pin_memory(), torch.cat(V, 1).cpu().pin_memory()


def _inputs(case, seed):
    """[(config, pos, vel)] of every instance."""
    dtype = torch.float64 if case.get("precision", "fp64") == "fp64" else torch.float32
    opt = {k: case[k] for k in ("mode", "subcells", "ntc_carry") if k in case}
    pin = lambda a: torch.from_numpy(np.ascontiguousarray(a)).to(dtype).pin_memory()  # noqa: E731
    out = []
    if case["kind"] == "relax":
        cfg, p, v = W.homogeneous_box(case["n"], case["kn"], seed=seed, n_steady=0)
        out.append((cfg, pin(p), pin(v)))
    elif case["kind"] == "ensemble":
        for i, (n, kn) in enumerate(zip(*_sizes(case))):
            s = (seed * 1009 + i) % (1 << 31)
            if i % 2 == 0:
                cfg, regions = W.sod(ncell=max(2, int(round(2 * n / 112.5))), ppc_left=100.0, lam_left=float(kn),
                                     n_steady=0)
                p, v = _particles(cfg, regions, s, dtype)
                out.append((dict(cfg, seed=s), p, v))
            else:
                cfg, p, v = W.homogeneous_box(int(n), float(kn), seed=s, n_steady=0)
                out.append((cfg, pin(p), pin(v)))
    else:
        cfg, regions = _flow(case)
        p, v = _particles(cfg, regions, seed, dtype)
        out.append((dict(cfg, seed=seed), p, v))
    return [(dict(c, **opt), p, v) for c, p, v in out]


def _sim(case, inputs):
    M = sum(v.shape[1] for _, _, v in inputs)
    open_box = case["kind"] not in ("relax", "sod", "ensemble")
    grow = 3.0 if case["kind"] == "jet" else 1.5
    cap = int(grow * M) + 200000 if open_box else M + 1024
    if case["kind"] == "jet":  # the orifice fills an empty domain: room for the developed jet
        cap = max(cap, int(case["ppc"] * (512 * case["scale"]) ** 2 * 0.12) + 200000)
    return sp.Sim([c for c, _, _ in inputs], PREC[case.get("precision", "fp64")], capacity=cap)


def _set(sim, inputs):
    for i, (_, p, v) in enumerate(inputs):
        put = sim.set_particles_ptr_f32 if p.dtype == torch.float32 else sim.set_particles_ptr
        put(i, p.data_ptr(), v.data_ptr(), v.shape[1])


def _tuned(case, inputs):
    """The collision schedule of a developed flow of this case, tuned once."""
    key = tuple(sorted((k, v) for k, v in case.items() if k not in ("name", "steps", "read")))
    if key not in _schedule:
        sim = _sim(case, inputs)
        _set(sim, inputs)
        sim.step(case["develop"])
        _schedule[key] = sim.autotune(steps_per_trial=5)
        sim.close()
    return _schedule[key]


def prepare(case, seed):
    if case["kind"] == "sort":
        nx, ny, n = case["nx"], case["ny"], case["keys"]
        g = torch.Generator(device="cuda")
        g.manual_seed(seed)
        r = lambda: torch.rand(n, generator=g, device="cuda")  # noqa: E731
        # the state was in cell order; one step moves a third of the
        # particles to a neighbouring cell, and a few leave (key 0xFFFFFFFF)
        cell = torch.sort((r().double() ** 1.5 * (nx * ny)).long()).values
        x, y = cell % nx, cell // nx
        a, b, c = r(), r(), r()
        x = (x + (a < 0.15).long() - (a > 0.9).long()).clamp(0, nx - 1)
        y = (y + (b < 0.08).long() - (b > 0.92).long()).clamp(0, ny - 1)
        key = torch.where(c < 0.002, torch.full_like(x, -1), x + nx * y).to(torch.int32)
        return {"case": case, "key": key, "start": torch.zeros(nx * ny + 1, dtype=torch.int32, device="cuda"),
                "perm": torch.zeros(n, dtype=torch.int32, device="cuda")}
    inputs = _inputs(case, seed)
    sched = _tuned(case, inputs) if case.get("tune") else None
    sim = _sim(case, inputs)
    st = {"case": case, "sim": sim}
    if sched:
        sim.set_schedule(*sched)
    if case["kind"] == "upload":
        st["host"] = inputs
    else:
        _set(sim, inputs)
        sim.step(case["develop"])
        sim.sync()
        if case["kind"] == "restart":  # the developed particles, as a checkpoint holds them
            p, v, _ = sim.particles(0)
            dt = inputs[0][1].dtype
            st["host"] = [(inputs[0][0], torch.from_numpy(p).to(dt).pin_memory(), torch.from_numpy(v).to(dt).pin_memory())]
    st["fields"] = torch.zeros(NF * sum(sim.ncells), dtype=torch.float64).pin_memory()
    # one flow: its fields by name (their units differ); an ensemble's fields stay in one buffer
    st["out"] = (dict(zip(sp.FIELDS, st["fields"].view(NF, -1).unbind(0))) if len(sim.ncells) == 1
                 else {"fields": st["fields"]})
    return st


def run(st):
    case = st["case"]
    if case["kind"] == "sort":
        sp.sort_cells_static(st["key"].data_ptr(), case["keys"], case["nx"] * case["ny"], st["start"].data_ptr(),
                             st["perm"].data_ptr())
        return {"start": st["start"], "perm": st["perm"]}
    sim = st["sim"]
    if "host" in st:
        _set(sim, st["host"])
    if case["kind"] != "upload":
        sim.step(case["steps"])
    at = st["fields"].data_ptr()
    for i, nc in enumerate(sim.ncells):
        sim.moments_into(i, 1 if case.get("read") == "mean" else 0, at)
        at += 8 * NF * nc
    out = dict(st["out"])
    if case["kind"] == "relax":  # an adaptive program reads the step that comes next
        out["dt"] = sim.dt(0)
    if sim.cfgs[0].get("n_surf", 0) and case.get("read") == "mean":
        tallies, out["time"] = sim.surface(0)
        out["surface"] = list(tallies)
    return out


def _count(case):
    """(particles, cells, dimensions) of a case, from its sizes alone."""
    k = case["kind"]
    if k == "relax":
        return case["n"], max(1, round(case["n"] / 56.25)), 1
    if k == "sod":
        return 0.5625 * case["cells"] * case["ppc"], case["cells"], 1
    if k == "ensemble":
        n = _sizes(case)[0]
        return float(n.sum()), float(n.sum()) / 56.25, 1
    if k in ("cylinder", "restart"):
        nc = round(600 * case["scale"]) * round(300 * case["scale"])
        return nc * case["ppc"], nc, 2
    if k == "jet":  # the steady jet: the orifice's flux through every station
        nc = max(8, round(512 * case["scale"])) ** 2
        return nc * case["ppc"] / 16, nc, 2
    if k in ("sphere", "upload"):
        nc = math.prod(round(v * case["scale"]) for v in (256, 128, 128))
        return nc * case["ppc"], nc, 3
    return case["nr"] * case["nt"] * case["ppc"], case["nr"] * case["nt"], 2


def work(case):
    if case["kind"] == "sort":
        return {"bytes": 8.0 * case["keys"] + 4.0 * case["nx"] * case["ny"], "flops": 0.0}
    M, nc, dim = _count(case)
    w = 8 if case.get("precision", "fp64") == "fp64" else 4
    state = w * (dim + 3) * M
    fields = 8.0 * NF * nc
    if case["kind"] == "upload":
        return {"bytes": state + fields, "flops": 20.0 * M}
    # per step: the state read and written once, the new cell of each
    # particle written and read once; about 60 operations per particle
    # (moments 20, collisions 20, flight and indexing 20)
    host = state if case["kind"] == "restart" else 0.0
    return {"bytes": case["steps"] * (2 * state + 8.0 * M) + fields + host, "flops": 60.0 * case["steps"] * M}


def exact(case, seed):
    """The moments of an uploaded state, in 64 bits; the sorted keys; no value for a stochastic step."""
    if case["kind"] == "sort":
        st = prepare(case, seed)
        key = st["key"].long()
        nc = case["nx"] * case["ny"]
        kept = key >= 0
        order = torch.sort(torch.where(kept, key, torch.full_like(key, nc)), stable=True).indices.int()
        m = int(kept.sum())
        perm = torch.zeros(case["keys"], dtype=torch.int32, device="cuda")
        perm[:m] = order[:m]
        start = torch.zeros(nc + 1, dtype=torch.int32, device="cuda")
        start[1:] = torch.cumsum(torch.bincount(key[kept], minlength=nc), 0).int()
        return {"start": start, "perm": perm}
    if case["kind"] != "upload":
        return None
    cfg, p, v = _inputs(case, seed)[0]
    x, c = p.numpy(), v.numpy()
    n = cfg["n"]
    idx = [np.clip(np.floor((x[d] - cfg["lo"][d]) * (n[d] / (cfg["hi"][d] - cfg["lo"][d]))), 0, n[d] - 1).astype(np.int64)
           for d in range(3)]
    cell = idx[0] + n[0] * (idx[1] + n[1] * idx[2])
    nc = n[0] * n[1] * n[2]
    total = lambda w: np.bincount(cell, weights=w, minlength=nc)  # noqa: E731
    N = np.bincount(cell, minlength=nc).astype(np.float64)
    f = np.zeros((NF, nc))
    with np.errstate(divide="ignore", invalid="ignore"):
        U = np.stack([np.where(N > 0, total(c[d]) / N, 0.0) for d in range(3)])
        C = c - U[:, cell]
        c2 = (C * C).sum(0)
        f[0], f[1] = N, N * cfg["Fn"] / cfg["cell_volume"]
        f[2:5] = U
        f[5] = np.where(N >= 2, total(c2) / (3.0 * cfg["R"] * (N - 1)), 0.0)
        for d in range(3):
            f[6 + d] = np.where(N >= 3, 0.5 * N / ((N - 1) * (N - 2)) * total(c2 * C[d]), 0.0)
        T, um = f[5], np.sqrt((U * U).sum(0))
        hot = (N >= 2) & (T > 0)
        f[9] = np.where(hot, cfg["mu_ref"] * (T / cfg["T_ref"]) ** cfg["omega"] / (f[1] * cfg["m"] * cfg["R"] * T), np.inf)
        L = min(W.cell_size(cfg))
        f[10] = np.where(hot, L / (um + np.sqrt(cfg["gamma"] * cfg["R"] * T)), np.where((N >= 2) & (um > 0), L / um, np.inf))
        f[11] = np.where(hot & (f[10] > f[9]), f[9] / f[10], 1.0)
    return dict(zip(sp.FIELDS, f))
