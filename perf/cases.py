"""The calls whose time matters to a user of the framework.

A host model hands the solver the state and the environment of its grid cells
once per chemistry step and takes the new state back (camp.Mechanism.solve and
its relatives).  The cases below are such steps over the range of mechanisms,
cell counts and options that this repository's workloads, tests and benchmark
use: one cell to a whole uneven domain, a gas mechanism, a sectional aerosol,
aerosol water as a parameter of the state, particle-resolved cells, the mixed
and the all-FP64 form, device and host buffers.  All draw synthetic cells of
`workloads.py` from the seed, at the tolerances used everywhere (rtol 1e-4,
atol 1e-5 ppb).
"""
import json
import math

import numpy as np
import torch

from paper_2111_07436_gb300 import camp, workloads

RTOL, ATOL = 1e-4, 1e-5

# Newton iterations and Jacobian setups of one cell over one call (means over
# the workloads' cells at their default step): the operations a solve at these
# tolerances takes are these counts times the operations of each part.
NEWTON = {"small": 10.8, "gas": 315.0, "multiphase": 346.0, "water": 462.0, "particles": 133.0, "arrow": 81.0}
SETUPS = {"small": 3.9, "gas": 25.0, "multiphase": 31.5, "water": 38.0, "particles": 16.0, "arrow": 12.4}


def listed():
    return [
        # a box model: one cell of 8 species, an hour of 60-s steps, every
        # step's state kept (latency alone)
        {"name": "box-hour", "call": "sequence", "mech": "small", "cells": 1, "dt": 60.0, "steps": 60, "fp64": False},
        # the smallest chunk of the request stream, one gas step
        {"name": "gas-chunk-256", "call": "solve", "mech": "gas", "species": 72, "cells": 256, "dt": 300.0, "fp64": False},
        # a domain of gas-phase chemistry, in both forms
        {"name": "gas-16384", "call": "solve", "mech": "gas", "species": 72, "cells": 16384, "dt": 180.0, "fp64": False},
        {"name": "gas-fp64-4099", "call": "solve", "mech": "gas", "species": 72, "cells": 4099, "dt": 180.0, "fp64": True},
        # gas and eight aerosol sections, in both forms
        {"name": "multiphase-4096", "call": "solve", "mech": "multiphase", "sections": 8, "cells": 4096, "dt": 300.0, "fp64": False},
        {"name": "multiphase-fp64-2047", "call": "solve", "mech": "multiphase", "sections": 8, "cells": 2047, "dt": 300.0, "fp64": True},
        # the same with aerosol water that follows the electrolytes
        {"name": "water-4096", "call": "solve", "mech": "water", "sections": 8, "cells": 4096, "dt": 300.0, "fp64": False},
        # particle-resolved cells: 128 particles (914 species) and the 10^4
        # particles of a box model (70018 species; the block-arrow solve)
        {"name": "particles-128x2048", "call": "solve", "mech": "particles", "particles": 128, "cells": 2048, "dt": 180.0, "fp64": False},
        {"name": "particles-10000x152", "call": "solve", "mech": "particles", "particles": 10000, "cells": 152, "dt": 180.0, "fp64": False},
        # a domain of uneven stiffness, half of it dark, a tenth cloudy: two
        # mechanisms in one call (the benchmark's default)
        {"name": "uneven-131072", "call": "batch", "mech": "uneven", "cells": 131072, "dt": 180.0, "fp64": False},
        # a host model that keeps its arrays in host memory: the whole call,
        # copies included, on a ragged chunk
        {"name": "gas-host-3001", "call": "host", "mech": "gas", "species": 72, "cells": 3001, "dt": 180.0, "fp64": False},
        # f(y) alone, for a host model's own integrator
        {"name": "forcing-65536", "call": "forcing", "mech": "gas", "species": 72, "cells": 65536, "dt": 0.0, "fp64": True},
    ]


def _logint(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more case: sizes log-uniform over the range of each kind."""
    kind = rng.choice(["small", "gas", "gas", "gas", "multiphase", "multiphase", "water", "particles", "arrow",
                       "uneven", "host", "forcing"])
    fp64 = rng.random() < 0.3
    dt = round(rng.uniform(60.0, 600.0), 1)
    if kind == "small":
        return {"call": "sequence", "mech": "small", "cells": _logint(rng, 1, 64), "dt": round(rng.uniform(30.0, 120.0), 1),
                "steps": rng.randint(10, 60), "fp64": fp64}
    if kind == "gas":
        return {"call": "solve", "mech": "gas", "species": rng.choice([rng.randint(24, 128), 72]),
                "cells": _logint(rng, 64, 16384), "dt": dt, "fp64": fp64}
    if kind == "multiphase" or kind == "water":
        return {"call": "solve", "mech": kind, "sections": rng.randint(1, 8), "cells": _logint(rng, 32, 4096), "dt": dt,
                "fp64": fp64}
    if kind == "particles":
        return {"call": "solve", "mech": "particles", "particles": _logint(rng, 20, 256), "cells": _logint(rng, 16, 1024),
                "dt": dt, "fp64": fp64}
    if kind == "arrow":
        return {"call": "solve", "mech": "particles", "particles": _logint(rng, 400, 10000), "cells": _logint(rng, 1, 152),
                "dt": round(rng.uniform(60.0, 180.0), 1), "fp64": fp64}
    if kind == "uneven":
        return {"call": "batch", "mech": "uneven", "cells": _logint(rng, 512, 65536), "dt": dt, "fp64": False}
    if kind == "host":
        return {"call": "host", "mech": "gas", "species": 72, "cells": _logint(rng, 64, 8192), "dt": dt, "fp64": fp64}
    return {"call": "forcing", "mech": "gas", "species": rng.choice([rng.randint(24, 128), 72]),
            "cells": _logint(rng, 256, 65536), "dt": 0.0, "fp64": True}


# ---- mechanisms and cells ------------------------------------------------------

def _gas(n):
    """The 72-species mechanism, or one of n species with reactions in the same proportions."""
    if n == 72:
        return workloads.large_gas_mechanism()
    part = [max(1, round(k * n / 72)) for k in (112, 28, 28, 9, 9)]
    return workloads.gas_mechanism(f"gas-{n}", n, *part, seed=1000 + n)


def _mechanism(case):
    kind = case["mech"]
    if kind == "small":
        return workloads.small_gas_mechanism()
    if kind == "gas":
        return _gas(case["species"])
    if kind == "particles":
        return workloads.particle_resolved_mechanism(case["particles"])
    m = workloads.water_mechanism() if kind == "water" else workloads.multiphase_mechanism()
    m["aerosol"]["sections"] = case["sections"]
    return m


def _groups(case, seed):
    """[(mechanism, state, env), ...] of the case: host arrays made from the seed."""
    if case["mech"] == "uneven":
        cloudy = case["cells"] // 10
        gas, clouds = workloads.large_gas_mechanism(), workloads.multiphase_mechanism()
        return [(gas, *workloads.cells(gas, case["cells"] - cloudy, seed=1000003 + 7 * seed, night_fraction=0.5)),
                (clouds, *workloads.cells(clouds, cloudy, seed=1000004 + 7 * seed, night_fraction=0.5,
                                          cloud_fraction=1.0))]
    m = _mechanism(case)
    fixed = dict(T=298.0, P=101300.0, sza=False) if case["mech"] == "small" and case["cells"] == 1 else {}
    return [(m, *workloads.cells(m, case["cells"], seed=2000003 + 7 * seed, **fixed))]


def prepare(case, seed):
    """The host model's side: compiled mechanisms, the cells' state and
    environment (device arrays; pinned host arrays for the host call), and the
    arrays that the call writes."""
    host = case["call"] == "host"
    place = (lambda a: torch.from_numpy(a).pin_memory()) if host else (lambda a: torch.from_numpy(a).cuda())
    s = {"case": dict(case), "variant": camp.VARIANT_FP64 if case["fp64"] else camp.VARIANT_MIXED, "groups": []}
    for m, y, env in _groups(case, seed):
        y, env = np.ascontiguousarray(y), np.ascontiguousarray(env)
        g = {"mech": camp.Mechanism(json.dumps(m)), "y0": place(y), "env": place(env)}
        g["state"] = g["y0"].clone().pin_memory() if host else g["y0"].clone()
        if not host:
            g["status"] = torch.zeros(len(y), dtype=torch.int32, device="cuda")
            g["atol"] = torch.tensor([ATOL], dtype=torch.float64, device="cuda")
            g["workspace"] = camp.workspace("cuda")
        if case["call"] == "sequence":
            g["trajectory"] = torch.zeros((case["steps"], *y.shape), dtype=torch.float64, device="cuda")
        s["groups"].append(g)
    return s


def run(s):
    """One chemistry step of every cell, from the state the host model hands over."""
    case, groups = s["case"], s["groups"]
    call, g = case["call"], groups[0]
    if call == "forcing":
        return g["mech"].forcing(g["y0"], g["env"])
    for q in groups:
        q["state"].copy_(q["y0"])
    if call == "host":
        status = g["mech"].solve_host(g["state"], g["env"], case["dt"], RTOL, ATOL, variant=s["variant"])
        return {"state": g["state"], "status": status}
    if call == "batch":
        camp.solve_batch(groups, case["dt"], RTOL, variant=s["variant"])
    elif call == "sequence":
        g["mech"].solve_sequence(g["state"], g["env"], case["dt"], case["steps"], RTOL, g["atol"],
                                 trajectory=g["trajectory"], status=g["status"], variant=s["variant"])
        return {"state": g["state"], "status": g["status"], "trajectory": g["trajectory"]}
    else:
        g["mech"].solve(g["state"], g["env"], case["dt"], RTOL, g["atol"], status=g["status"], variant=s["variant"],
                        workspace=g["workspace"])
    return [{"state": q["state"], "status": q["status"]} for q in groups]


def work(case):
    """Bytes: state and environment in, state, status and trajectory out.
    Operations: the mean counts above times those of one f, one triangular
    solve, one Jacobian and one factorisation of the compiled mechanism."""
    if case["mech"] == "uneven":
        cloudy = case["cells"] // 10
        parts = [({"call": "solve", "mech": "gas", "species": 72, "cells": case["cells"] - cloudy}, "gas"),
                 ({"call": "solve", "mech": "multiphase", "sections": 8, "cells": cloudy}, "multiphase")]
    else:
        parts = [(case, case["mech"])]
    nbytes = flops = 0.0
    for c, kind in parts:
        i = camp.Mechanism(json.dumps(_mechanism(c)), device=False).info
        if i.block_arrow:
            kind = "arrow"
        if c["call"] == "forcing":
            nbytes += 8.0 * c["cells"] * (2 * i.n_species + i.n_env)
            flops += float(c["cells"]) * i.flops_forcing
            continue
        outs = 1 + c.get("steps", 1) if c["call"] == "sequence" else 1
        nbytes += c["cells"] * (8.0 * (i.n_species * (1 + outs) + i.n_env) + 4)
        flops += c["cells"] * c.get("steps", 1) * (NEWTON[kind] * (i.flops_forcing + i.flops_solve + 8 * i.n_species) +
                                                   SETUPS[kind] * (i.flops_jacobian + i.flops_factor))
    return {"bytes": nbytes, "flops": flops}


# ---- f(y) in plain numpy ---------------------------------------------------------

KB = 1.380649e-23  # J/K


def _arr300(r, key, T):
    return r[key + "_A"] * np.exp(r[key + "_C"] / T) * (T / 300.0) ** r[key + "_B"]


def _forcing(mech, y, env):
    """f(y) [ppb/s] of a gas mechanism, reaction by reaction."""
    idx = {s["name"]: k for k, s in enumerate(mech["species"])}
    T, P = env[:, 0], env[:, 1]
    M = P / (KB * T) * 1e-6  # molec/cm^3
    f, slot = np.zeros_like(y), 2
    for r in mech["reactions"]:
        t = r["type"]
        if t in ("EMISSION", "FIRST_ORDER_LOSS"):
            k, i = env[:, slot], idx[r["species"]]
            slot += 1
            f[:, i] += k if t == "EMISSION" else -k * y[:, i]
            continue
        if t == "PHOTOLYSIS":
            k = env[:, slot]
            slot += 1
        elif t == "ARRHENIUS":
            k = r["A"] * np.exp(r["C"] / T) * (T / r["D"]) ** r["B"] * (1.0 + r["E"] * P)
        else:
            k0M, kinf = _arr300(r, "k0", T) * M, _arr300(r, "kinf", T)
            x = k0M / kinf
            k = k0M / (1.0 + x) * r["Fc"] ** (1.0 / (1.0 + (np.log10(x) / r["N"]) ** 2))
        if t != "PHOTOLYSIS":
            k = k * (M * 1e-9) ** (sum(r["reactants"].values()) - 1)
        rate = k.copy()
        for a, m in r["reactants"].items():
            rate *= y[:, idx[a]] ** m
        for a, m in r["reactants"].items():
            f[:, idx[a]] -= m * rate
        for a, v in r["products"].items():
            f[:, idx[a]] += v * rate
    return f


def exact(case, seed):
    """f(y) in 64 bits.  A whole solve has none: an adaptive integration of
    every cell to 64-bit accuracy takes minutes in numpy."""
    if case["call"] != "forcing":
        return None
    (mech, y, env), = _groups(case, seed)
    return _forcing(mech, y, env)
