"""Timed cases of the public entry points: what a program that uses the library has it do.

Four ways of use, over the sizes and chemistries of the tests, the benchmark and the serving mix:

  run       one mesh handle with its model: counts in, ``rdsplit_run`` over some periods, counts out
  static    the allocation-free ``rdsplit_run_static`` on the caller's device arrays
  ensemble  many handles advanced together by ``rdsplit_ensemble_run``
  serve     requests in host memory through ``serving.Server`` (mesh and model upload, continuous
            batching, results back on the host)

Meshes are kept per case (a program builds its mesh once); the seed decides the initial counts and the
random streams.  Every output is a whole number.
"""
from __future__ import annotations

import functools
import math

import numpy as np
import torch

from paper_1512_03126_gb300 import inputs as I
from paper_1512_03126_gb300 import rdsplit as rd
from paper_1512_03126_gb300 import serving


def listed():
    return [
        # the smallest call: a recording loop reads the counts every few periods (the 960-tet tube
        # with influx at its ends)
        {"name": "tube_readout", "kind": "run", "mesh": "box", "nx": 2, "ny": 2, "nz": 40, "h": 1e-7,
         "model": "influx", "S": 1, "conc": 5.0, "periods": 8, "rule": 0, "shuffled": False},
        # the 3,072-tet diffusion cube from its point source over its whole run
        {"name": "cube_3072_point", "kind": "run", "mesh": "box", "nx": 8, "ny": 8, "nz": 8, "h": 1.25e-7,
         "model": "diffusion", "S": 1, "conc": 0.0, "periods": 217, "rule": 0, "shuffled": False},
        # surface diffusion with first-order decay on a triangle sheet
        {"name": "sheet_decay", "kind": "run", "mesh": "sheet", "nx": 61, "ny": 47, "nz": 1, "h": 1e-7,
         "model": "decay", "S": 1, "conc": 7.0, "periods": 120, "rule": 0, "shuffled": False},
        # the 48,000-tet A/B/C reaction-diffusion cube, its first periods
        {"name": "abc_48000", "kind": "run", "mesh": "box", "nx": 20, "ny": 20, "nz": 20, "h": 1e-7,
         "model": "abc", "S": 3, "conc": 10.0, "periods": 200, "rule": 0, "shuffled": False},
        # a random chemistry of six species on a box of uneven sides
        {"name": "random6_ragged", "kind": "run", "mesh": "box", "nx": 23, "ny": 17, "nz": 29, "h": 5e-8,
         "model": "random", "S": 6, "conc": 20.0, "periods": 100, "rule": 0, "shuffled": False},
        # a random chemistry of eleven species (30 reactions), under the half-step transfer rule
        {"name": "random11_mid", "kind": "run", "mesh": "box", "nx": 11, "ny": 13, "nz": 15, "h": 8e-8,
         "model": "random", "S": 11, "conc": 5.0, "periods": 60, "rule": 2, "shuffled": False},
        # a mesh generator's unordered numbering, stored along the curve: the largest diffusion cube
        {"name": "cube_384000_reordered", "kind": "run", "mesh": "box", "nx": 40, "ny": 40, "nz": 40, "h": 2.5e-8,
         "model": "diffusion", "S": 1, "conc": 10.0, "periods": 100, "rule": 0, "shuffled": True},
        # the long bar: 2.4 M tets, 8 species, 14 masked reactions
        {"name": "bar_2400000", "kind": "run", "mesh": "box", "nx": 20, "ny": 20, "nz": 1000, "h": 5e-8,
         "model": "bar", "S": 8, "conc": 0.0, "periods": 24, "rule": 0, "shuffled": False},
        # a plugin's step on its own memory: coarse tets that hold tens of molecules
        {"name": "static_abc", "kind": "static", "mesh": "box", "nx": 9, "ny": 10, "nz": 11, "h": 2e-7,
         "model": "abc", "S": 3, "conc": 20.0, "periods": 40, "rule": 0, "shuffled": False},
        # cubes of many sizes from their point sources, as in the batched ensemble
        {"name": "ensemble_cubes", "kind": "ensemble", "n_sims": 40, "n_lo": 6, "n_hi": 24, "model": "diffusion",
         "conc": 0.0, "t_end": 0.02},
        # realisations of one small tube: means and variances over seeds
        {"name": "ensemble_tubes", "kind": "ensemble", "n_sims": 152, "n_lo": 0, "n_hi": 0, "model": "influx",
         "conc": 0.0, "t_end": 0.05},
        # the serving mix: random chemistries of 1..8 species, sizes log-uniform
        {"name": "serve_mix", "kind": "serve", "n_requests": 24, "n_lo": 6, "n_hi": 32, "t_hi": 0.01, "cluster": 8},
    ]


def draw(rng):
    kind = rng.choices(["run", "static", "ensemble", "serve"], [8, 1, 2, 1])[0]
    if kind == "ensemble":
        hi = rng.randint(8, 24)
        tubes = rng.random() < 0.3
        return {"kind": kind, "n_sims": rng.randint(3, 96 if tubes else 40), "n_lo": 0 if tubes else rng.randint(3, 6),
                "n_hi": 0 if tubes else hi, "model": "influx" if tubes else rng.choice(["diffusion", "abc"]),
                "conc": 0.0 if tubes else _log(rng, 0.2, 20.0),
                "t_end": _log(rng, 0.01, 0.05) if tubes else _log(rng, 0.001, 0.01)}
    if kind == "serve":
        return {"kind": kind, "n_requests": rng.randint(4, 24), "n_lo": 6, "n_hi": rng.randint(10, 32),
                "t_hi": _log(rng, 0.002, 0.01), "cluster": rng.choice([2, 4, 8])}
    model = rng.choice(["diffusion", "abc", "random", "random", "bar", "decay", "influx"])
    S = {"abc": 3, "bar": 8, "random": rng.randint(2, 11)}.get(model) or rng.choice([1, 1, 2, 4, 16])
    if model in ("influx", "decay"):
        S = 1
    cells = _log(rng, 20, 5e3 if kind == "static" else 1.2e5 if model == "diffusion" else 8e4)
    side = cells ** (1.0 / 3.0)
    nx = max(1, round(side * rng.uniform(0.5, 1.1)))
    ny = max(1, round(side * rng.uniform(0.6, 1.3)))
    nz = max(2, round(cells / (nx * ny)))
    mesh = "sheet" if model == "decay" and kind == "run" else "box"
    if mesh == "sheet":
        nx, ny, nz = rng.randint(5, 90), rng.randint(5, 90), 1
    T = 6 * nx * ny * nz
    cap = 1.5e8 / (T * S)
    return {"kind": kind, "mesh": mesh, "nx": nx, "ny": ny, "nz": nz, "h": _log(rng, 3e-8, 2e-7), "model": model,
            "S": S, "conc": _log(rng, 0.5, 30.0), "periods": max(2, min(round(_log(rng, 4, 200)), int(cap))),
            "rule": rng.choice([0, 0, 0, 1, 2]) if kind == "run" else 0,
            "shuffled": mesh == "box" and kind == "run" and rng.random() < 0.25}


def _log(rng, lo, hi):
    return float("%.3g" % math.exp(rng.uniform(math.log(lo), math.log(hi))))


@functools.lru_cache(maxsize=128)
def _box(nx, ny, nz, h, mesh_seed, shuffled):
    mesh = I.kuhn_box(nx, ny, nz, (nx * h, ny * h, nz * h), 0.2, mesh_seed)
    return I.shuffle_mesh(mesh, mesh_seed)[0] if shuffled else mesh


@functools.lru_cache(maxsize=8)
def _sheet(nx, ny, h):
    return I.triangle_sheet(nx, ny, (nx * h, ny * h), 0.2, 31)


def _mesh_of(case):
    if case["mesh"] == "sheet":
        return _sheet(case["nx"], case["ny"], case["h"])
    return _box(case["nx"], case["ny"], case["nz"], case["h"], 4, case["shuffled"])


def _tau_guess(mesh, D):
    """The period of the method's definition, 1 / max(D * sum of A / (V dist)), for rates given per period."""
    with np.errstate(divide="ignore", invalid="ignore"):
        g = np.where(mesh.adj >= 0, mesh.area / (mesh.vol[:, None] * mesh.dist), 0.0)
    top = float(np.max(np.sum(g, axis=1)) * np.max(D))
    return 1.0 / top if top > 0 else 1.0


def _influx_model(mesh):
    """Zero-order influx of about four molecules per period into the tets of the two end layers along z."""
    D = np.array([1e-12])
    per_s = 4.0 / _tau_guess(mesh, D)
    k = np.array([per_s / (I.AVOGADRO * 1e3 * float(np.mean(mesh.vol)))])
    L, layer = mesh.size[2], mesh.size[2] / max(1, mesh.shape[2])
    ends = (mesh.centroid[:, 2] < layer) | (mesh.centroid[:, 2] > L - layer)
    return I.Model(D=D, lhs=np.zeros((1, 1), np.int32), rhs=np.ones((1, 1), np.int32), k=k,
                   mask=ends.astype(np.uint8)[None, :], names=["A"])


def _model_of(kind, mesh, S):
    if kind == "abc":
        return I.abc_model()
    if kind == "bar":
        return I.bar_model(mesh)
    if kind == "random":
        return I.random_model(mesh, S, np.random.Generator(np.random.PCG64(9000 + S)))
    if kind == "influx":
        return _influx_model(mesh)
    if kind == "decay":
        return I.Model(D=np.array([0.5e-12]), lhs=np.ones((1, 1), np.int32), rhs=np.zeros((1, 1), np.int32),
                       k=np.array([20.0]), names=["A"])
    return I.diffusion_model(1e-12, S)


def _counts_of(case, mesh, model, seed):
    """Initial counts: a point source of 6,000, molecules per triangle, or concentrations (uM) by volume."""
    rng = np.random.Generator(np.random.PCG64(seed))
    T, S = mesh.n_tets, model.n_species
    counts = np.zeros((T, S), np.int32)
    if case["model"] == "bar":
        V = float(np.sum(mesh.vol))
        free, buf = I.molecules(0.1e-6, V), I.molecules(50e-6, V)
        return I.place_by_volume(mesh, [free, free, free, buf, buf, 0, 0, 0], seed)
    if case["model"] == "decay":
        return rng.poisson(case["conc"], (T, 1)).astype(np.int32)
    if case["model"] == "diffusion":
        counts[int(rng.integers(T)), 0] = 6000
    if case["conc"] > 0.0:
        n = I.molecules(case["conc"] * 1e-6, float(np.sum(mesh.vol)))
        totals = [n, n, 0] if case["model"] == "abc" else [n] * S
        counts += I.place_by_volume(mesh, totals, seed)
    return counts


def _sizes(case):
    return [case["n_lo"] + (i * 7919 + 3) % (case["n_hi"] - case["n_lo"] + 1) for i in range(case["n_sims"])]


def _requests(case):
    """Sizes log-uniform, 1..8 species, end times uniform: the serving mix's draws, fixed per case."""
    rng = np.random.Generator(np.random.PCG64(5))
    out = []
    for i in range(case["n_requests"]):
        n = int(round(math.exp(rng.uniform(math.log(case["n_lo"]), math.log(case["n_hi"])))))
        out.append((n, int(rng.integers(1, 9)), float(rng.uniform(1e-3, case["t_hi"]))))
    return out


def prepare(case, seed):
    kind = case["kind"]
    if kind == "serve":
        requests, prepared = [], {}
        for i, (n, S, t_end) in enumerate(_requests(case)):
            mesh = _box(n, n, n, 5e-8, 5000 + i, False)
            model = I.random_model(mesh, S, np.random.Generator(np.random.PCG64(9000 + i)))
            free = I.molecules(1e-6, float(np.sum(mesh.vol)))
            counts = I.place_by_volume(mesh, [free] * S, 1000 * seed + i)
            requests.append(I.Request(i, 0.0, n, S, t_end, 9000 + i))
            prepared[i] = I.Workload("request", mesh, model, counts, t_end, 64 * seed + i)
        server = serving.Server(keep_counts=True, slice_work=20_000_000, cluster=case["cluster"])
        return {"kind": kind, "server": server, "requests": requests, "prepared": prepared}
    if kind == "ensemble":
        sims, counts, t_end, seeds = [], [], [], []
        for i in range(case["n_sims"]):
            if case["n_hi"] == 0:
                mesh = _box(2, 2, 40, 1e-7, 77, False)
            else:
                n = _sizes(case)[i]
                mesh = _box(n, n, n, 1e-6 / n, 1000 + i, False)
            model = _model_of(case["model"], mesh, 1)
            sims.append(rd.Simulation(mesh, model))
            counts.append(torch.from_numpy(_counts_of(case, mesh, model, 1000 * seed + i)).cuda())
            t_end.append(case["t_end"])
            seeds.append(1000 * seed + i)
        total = sum(c.numel() for c in counts)
        out = torch.empty(total, dtype=torch.int32, device="cuda")
        parts = torch.split(out, [c.numel() for c in counts])
        return {"kind": kind, "sims": sims, "counts": counts, "t_end": t_end, "seeds": seeds, "out": out,
                "parts": parts}
    mesh = _mesh_of(case)
    model = _model_of(case["model"], mesh, case["S"])
    counts = torch.from_numpy(_counts_of(case, mesh, model, seed)).cuda()
    # an end time between two periods: the last one is shortened to end on it
    t_end = (case["periods"] - 0.4) * _tau_guess(mesh, model.D)
    if kind == "static":
        def dev(a):
            return None if a is None else torch.from_numpy(np.ascontiguousarray(a)).cuda()
        return {"kind": kind, "n": mesh.n_tets, "adj": dev(mesh.adj), "vol": dev(mesh.vol), "area": dev(mesh.area),
                "dist": dev(mesh.dist), "mask": dev(model.mask), "model": model, "counts": counts, "t_end": t_end,
                "seed": seed}
    sim = rd.Simulation(mesh, model, rule=case["rule"], reorder=case["shuffled"])
    return {"kind": kind, "sim": sim, "counts": counts, "out": torch.empty_like(counts), "t_end": t_end, "seed": seed}


def run(state):
    kind = state["kind"]
    if kind == "run":
        h = state["sim"].h
        rd.rdsplit_set_counts_device(h, state["counts"])
        rd.rdsplit_set_time(h, 0.0, 0)
        rd.rdsplit_run(h, state["t_end"], state["seed"])
        rd.rdsplit_get_counts_device(h, state["out"])
        return {"counts": state["out"], "period": rd.rdsplit_get_time(h)[1]}
    if kind == "static":
        m = state["model"]
        counts = state["counts"].clone()
        _, period = rd.rdsplit_run_static(state["n"], state["adj"], state["vol"], state["area"], state["dist"],
                                          m.n_species, m.D, m.n_reactions, m.lhs, m.rhs, m.k, state["mask"],
                                          m.tau_scale, counts, 0.0, 0, state["t_end"], state["seed"])
        return {"counts": counts, "period": period}
    if kind == "ensemble":
        for sim, counts in zip(state["sims"], state["counts"]):
            rd.rdsplit_set_counts_device(sim.h, counts)
            rd.rdsplit_set_time(sim.h, 0.0, 0)
        rd.rdsplit_ensemble_run([s.h for s in state["sims"]], state["t_end"], state["seeds"])
        for sim, part in zip(state["sims"], state["parts"]):
            rd.rdsplit_get_counts_device(sim.h, part)
        return {"counts": state["out"]}
    records = state["server"].serve(state["requests"], state["prepared"])
    records = sorted(records, key=lambda r: r.rid)
    return {"counts": np.concatenate([r.counts.ravel() for r in records]),
            "tet_periods": np.array([r.tet_periods for r in records], np.int64)}


def exact(case, seed):
    """Counts are draws from the library's own random streams: whole numbers that have to stay equal, with no
    64-bit value beside them."""
    return None


def work(case):
    """Bytes: counts in and out, neighbours (16 B), face areas and distances (64 B) and volume (8 B) of every tet,
    once.  Operations: one uniform per molecule and period, a quarter of a Philox block of ten rounds (20
    operations)."""
    if case["kind"] == "serve":
        T = [6 * n ** 3 for n, _, _ in _requests(case)]
        size = sum(t * (88 + 8 * S) for t, (_, S, _) in zip(T, _requests(case)))
        moved = sum(t * S * 0.0125 * t_end / 1.5e-5 for t, (_, S, t_end) in zip(T, _requests(case)))
        return {"bytes": size, "flops": 20 * moved}
    if case["kind"] == "ensemble":
        if case["n_hi"] == 0:
            return {"bytes": case["n_sims"] * 960 * 96, "flops": 20 * case["n_sims"] * 96 * (case["t_end"] / 2e-4) ** 2}
        ns = _sizes(case)
        S = 3 if case["model"] == "abc" else 1
        per = [case["t_end"] / (0.025 / n ** 2) * (6000 + 1200 * case["conc"]) for n in ns]
        return {"bytes": sum(6 * n ** 3 * (88 + 8 * S) for n in ns), "flops": 20 * sum(per)}
    cells = case["nx"] * case["ny"] * case["nz"]
    T = (2 if case["mesh"] == "sheet" else 6) * cells
    per_tet = {"bar": 1.26, "decay": case["conc"]}.get(
        case["model"], case["conc"] * 602.2 * 1e18 * case["h"] ** 3 / 6 * (2 if case["model"] == "abc" else case["S"]))
    molecules = T * per_tet + (6000 if case["model"] == "diffusion" else 0)
    return {"bytes": T * (88 + 8 * case["S"]), "flops": 20 * molecules * case["periods"]}
