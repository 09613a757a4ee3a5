"""The work that users of the library have it do, as cases that can be timed.

Every case is one pass through the public entry points (the Python binding of
include/steps_gpu.h). Lengths are given in diffusion windows of the
simulation's own tau, as real numbers: the fraction is the shortened last
window that a run to an arbitrary end time has. Counts are integers drawn from
counter-based random numbers, so outputs are whole numbers and there is no
64-bit value to hold them against.

Kinds of case:

  run      a whole job through host buffers: set the initial counts, run to the
           end time, read the final counts (a parameter sweep, a seed study)
  noalloc  the same on counts that live on the device, through the entry point
           that allocates nothing (an application that couples the step to its
           own device code)
  record   a calcium-burst segment: the influx rate is set, the run records one
           species at a sample of the tets at fixed intervals into device
           memory, the final counts are read
  batch    replicates of several meshes advanced together, each with a seed of
           its own (statistics over repeated runs)
  served   jobs of mixed kinds and sizes, all queued at once, through the job
           server until the last result is taken
"""
from __future__ import annotations

import math
from functools import lru_cache

import numpy as np
import torch

from paper_1610_02258_gb300 import capi
from paper_1610_02258_gb300 import inputs as I

UM = I.UM
NET_SEED = 5           # reaction network of the box workloads
CUBOID_EDGE = 0.5      # um, cube edge of the cuboid workloads
DENDRITE_EDGE = 0.149  # um, voxel edge of the 1.03M-tet dendrite


def listed():
    return [
        # the smallest job: the 2 x 2 x 10 um cuboid (1,920 tets, A + B <-> C), 10 ms
        {"name": "cuboid-1920", "kind": "run", "family": "cuboid", "length": 20, "windows": 13.52},
        # the same chemistry on a longer cuboid, counts resident on the device
        {"name": "cuboid-noalloc", "kind": "noalloc", "family": "cuboid", "length": 104, "windows": 27.04},
        # the box of the benchmark network meshed coarsely: few tets, many molecules in each
        {"name": "box-coarse", "kind": "run", "family": "box", "across": 8, "nx": 80, "ny": 8, "nz": 8,
         "density": 1.0, "windows": 23.78, "law": "euler", "occupancy": "mean"},
        # the benchmark: 100 x 10 x 10 um, 294,780 tets, 10 species, 20 reactions, 20 ms
        {"name": "box", "kind": "run", "family": "box", "across": 17, "nx": 170, "ny": 17, "nz": 17,
         "density": 1.0, "windows": 98.52, "law": "euler", "occupancy": "mean"},
        # the density experiment's ends: a tenth and ten times the concentrations
        {"name": "box-sparse", "kind": "run", "family": "box", "across": 17, "nx": 170, "ny": 17, "nz": 17,
         "density": 0.1, "windows": 98.52, "law": "euler", "occupancy": "mean"},
        {"name": "box-dense", "kind": "run", "family": "box", "across": 17, "nx": 170, "ny": 17, "nz": 17,
         "density": 10.0, "windows": 98.52, "law": "euler", "occupancy": "mean"},
        # the mesh experiment's fine end: the same box with 26 cubes across (1.05M tets)
        {"name": "box-fine", "kind": "run", "family": "box", "across": 26, "nx": 260, "ny": 26, "nz": 26,
         "density": 1.0, "windows": 322.3, "law": "euler", "occupancy": "mean"},
        # an odd-sized box under the other leave law and the end-count trial rule
        {"name": "box-exp-end", "kind": "run", "family": "box", "across": 17, "nx": 71, "ny": 13, "nz": 19,
         "density": 2.5, "windows": 60.3, "law": "exp", "occupancy": "end"},
        # the 1.03M-tet dendrite with the 20-species calcium network, 2 ms
        {"name": "dendrite", "kind": "run", "family": "dendrite", "tets": 1030000, "windows": 609.0},
        # a burst segment on a coarser dendrite: 60 recordings of Ca at 1 % of the tets
        {"name": "dendrite-record", "kind": "record", "family": "dendrite", "tets": 300000, "windows": 366.0,
         "records": 60, "every": 100},
        # replicates: four meshes of 10k to 300k tets, six seeds of each
        {"name": "replicates", "kind": "batch", "members": 24, "meshes": 4, "lo": 10000, "hi": 300000,
         "windows": 98.52},
        # a burst of mixed jobs at the server
        {"name": "served-mix", "kind": "served", "jobs": 16, "lo": 2000, "hi": 200000, "mix": 21, "windows": 40.0},
    ]


# ---------------------------------------------------------------- drawn cases

def _logu(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


# Rough cost of a drawn run, in tet-windows weighted by the molecules in a
# tet, against the largest listed cases: only used to cut the window count.
COST_LIMIT = 2.5e8


def _windows(rng, lo, hi, tets, molecules_per_tet):
    weight = 0.4 + molecules_per_tet / 20.0
    most = max(lo, min(hi, COST_LIMIT / (tets * weight)))
    return round(_logu(rng, lo, most), 2)


def _draw_box(rng, law, occupancy):
    across = rng.randint(6, 26)
    ny, nz = rng.randint(5, 26), rng.randint(5, 26)
    tets = _logu(rng, 8e3, 1.05e6)
    nx = max(1, int(tets / (6 * ny * nz)))
    tets = 6 * nx * ny * nz
    per_tet = 404.0 * (10.0 / across) ** 3 / 6.0  # molecules per tet at the benchmark's densities
    density = round(_logu(rng, 0.1, max(0.2, min(10.0, 140.0 / per_tet))), 3)
    return {"kind": "run", "family": "box", "across": across, "nx": nx, "ny": ny, "nz": nz, "density": density,
            "windows": _windows(rng, 6.0, 320.0, tets, per_tet * density), "law": law, "occupancy": occupancy}


def draw(rng):
    kind = rng.choice(["cuboid", "cuboid", "box", "box", "box", "box", "box", "dendrite", "dendrite", "batch",
                       "served"])
    if kind == "cuboid":
        return {"kind": rng.choice(["run", "noalloc"]), "family": "cuboid", "length": int(_logu(rng, 10, 600)),
                "windows": round(_logu(rng, 4.0, 120.0), 2)}
    if kind == "box":
        return _draw_box(rng, rng.choice(["euler", "euler", "exp"]), rng.choice(["mean", "mean", "end"]))
    if kind == "dendrite":
        tets = int(_logu(rng, 2e4, 1.03e6))
        windows = _windows(rng, 30.0, 600.0, tets, 0.1)
        if rng.random() < 0.5:
            return {"kind": "run", "family": "dendrite", "tets": tets, "windows": windows}
        return {"kind": "record", "family": "dendrite", "tets": tets, "windows": windows,
                "records": rng.randint(2, 60), "every": int(_logu(rng, 20, 1000))}
    if kind == "batch":
        members = rng.randint(2, 24)
        return {"kind": "batch", "members": members, "meshes": rng.randint(1, min(4, members)),
                "lo": 10000, "hi": int(_logu(rng, 2e4, 3e5)), "windows": round(_logu(rng, 6.0, 98.52), 2)}
    return {"kind": "served", "jobs": rng.randint(2, 16), "lo": 2000, "hi": int(_logu(rng, 4e3, 2e5)),
            "mix": rng.randint(0, 10**6), "windows": round(_logu(rng, 8.0, 40.0), 1)}


# ---------------------------------------------------------------- workloads

class _Load:
    """Mesh, model, molecule totals and where they are placed."""

    def __init__(self, verts, tets, model, totals, subset=None, masks=None):
        self.verts, self.tets, self.model = verts, tets, model
        self.totals = totals          # molecules per species
        self.subset = subset or {}    # species -> tets it starts in (default: all)
        self.masks = masks or {}      # reaction -> active tets
        self.nt = int(tets.shape[0])

    def place(self, seed):
        """Initial counts [S, nt]: every molecule in a tet drawn uniformly."""
        rng = np.random.default_rng(seed)
        out = np.zeros((len(self.totals), self.nt), np.int32)
        for s, n in enumerate(self.totals):
            idx = self.subset.get(s)
            if idx is None:
                out[s] = np.bincount(rng.integers(0, self.nt, n), minlength=self.nt)
            else:
                out[s, idx] = np.bincount(rng.integers(0, len(idx), n), minlength=len(idx))
        return out


@lru_cache(maxsize=8)
def _cuboid(length):
    verts, tets = I.kuhn_box_mesh(4, 4, length, CUBOID_EDGE * UM)
    n = int(round(125.0 * 4.0 * length * CUBOID_EDGE))  # 125 A and 125 B per um^3
    return _Load(verts, tets, I.config1_model(), [n, n, 0])


@lru_cache(maxsize=8)
def _box(across, nx, ny, nz, density):
    h = 10.0 / across * UM
    verts, tets = I.kuhn_box_mesh(nx, ny, nz, h)
    verts = I.jitter_box_vertices(verts, h, 0.2, seed=1)
    model = I.random_network(NET_SEED)
    dens = np.random.default_rng(2).uniform(1.0, 100.0, size=model.n_species) * density  # per um^3
    vol = nx * ny * nz * (10.0 / across) ** 3
    return _Load(verts, tets, model, [int(round(d * vol)) for d in dens])


@lru_cache(maxsize=8)
def _dendrite(target):
    w = I.config3_scaled(target)
    soma = np.flatnonzero(next(iter(w.reac_masks.values())))
    ca = w.model.names.index("Ca")
    return _Load(w.verts, w.tets, w.model, [int(n) for n in w.counts.sum(axis=1)], {ca: soma}, w.reac_masks)


def _load(case):
    if case["family"] == "cuboid":
        return _cuboid(case["length"])
    if case["family"] == "box":
        return _box(case["across"], case["nx"], case["ny"], case["nz"], case["density"])
    return _dendrite(case["tets"])


def _simulation(load, seed, **options):
    sim = capi.Simulation(load.verts, load.tets, load.model, seed, **options)
    for r, mask in load.masks.items():
        sim.set_reac_mask(r, mask)
    return sim


def _box_lengths(case):
    """Cube counts along the box of the batch's meshes (17 x 17 cubes across)."""
    n = case["meshes"]
    sizes = [case["lo"] * (case["hi"] / case["lo"]) ** ((j + 0.5) / n) for j in range(n)]
    return [max(1, int(round(size / (6 * 17 * 17)))) for size in sizes]


def _jobs(case):
    """(family, size, windows) of the served jobs: sizes log-uniform, snapped to
    six prototypes per family; lengths log-uniform up to the case's windows."""
    rng = np.random.default_rng(case["mix"])
    grid = np.geomspace(case["lo"], case["hi"], 6)
    jobs = []
    for _ in range(case["jobs"]):
        family = ("cuboid", "box", "dendrite")[int(rng.integers(0, 3))]
        size = int(grid[int(rng.integers(0, 6))])
        jobs.append((family, size, round(float(case["windows"] * 8.0 ** -rng.uniform()), 2)))
    return jobs


def _job_load(family, size):
    if family == "cuboid":
        return _cuboid(max(1, int(round(size / 96))))
    if family == "box":
        return _box(17, max(1, int(round(size / (6 * 17 * 17)))), 17, 17, 1.0)
    return _dendrite(size)


# ---------------------------------------------------------------- one pass

def _pinned(counts):
    """A caller's page-locked copy of a count array."""
    return torch.from_numpy(counts).pin_memory().numpy()


def _result(load):
    return torch.empty((load.model.n_species, load.nt), dtype=torch.int32, pin_memory=True).numpy()


def prepare(case, seed):
    kind = case["kind"]
    if kind == "batch":
        loads = [_box(17, nx, 17, 17, 1.0) for nx in _box_lengths(case)]
        protos = [_simulation(load, seed) for load in loads]
        members, counts, results = [], [], []
        for j in range(case["members"]):
            q = j % case["meshes"]
            members.append(protos[q] if j < case["meshes"] else protos[q].clone(seed + 1000 + j))
            counts.append(_pinned(loads[q].place(seed + 1000 + j)))
            results.append(_result(loads[q]))
        return {"kind": kind, "sims": members, "batch": capi.Batch(members), "counts": counts, "results": results,
                "length": case["windows"] * protos[0].tau}
    if kind == "served":
        protos, jobs = {}, []
        for j, (family, size, windows) in enumerate(_jobs(case)):
            load = _job_load(family, size)
            if (family, size) not in protos:
                protos[family, size] = _simulation(load, 1, specialize=1)
            proto = protos[family, size]
            jobs.append((proto, seed + 1000 + j, load.place(seed + 1000 + j), windows * proto.tau))
        return {"kind": kind, "jobs": jobs, "protos": protos,
                "server": capi.NativeServer(max_jobs=128, wave_windows=32, specialize=1)}
    load = _load(case)
    options = {}
    if case["family"] == "box":
        options["leave_law"] = capi.STEPS_LEAVE_EXP if case["law"] == "exp" else capi.STEPS_LEAVE_EULER
        options["occupancy"] = capi.STEPS_OCC_END if case["occupancy"] == "end" else capi.STEPS_OCC_MEAN
    sim = _simulation(load, seed, **options)
    state = {"kind": kind, "sim": sim, "counts": _pinned(load.place(seed)), "length": case["windows"] * sim.tau}
    if kind == "noalloc":
        state["initial"] = torch.from_numpy(state["counts"]).cuda()
        state["work"] = torch.empty_like(state["initial"])
        return state
    state["result"] = _result(load)
    if kind == "record":
        tets = np.sort(np.random.default_rng(seed).choice(load.nt, max(1, load.nt // case["every"]), replace=False))
        state["species"] = np.array([load.model.names.index("Ca")], np.int32)
        state["tets"] = tets.astype(np.int32)
        state["every"] = state["length"] / case["records"]
        state["records"] = torch.zeros((case["records"] + 1, 1, tets.size), dtype=torch.int32, device="cuda")
        state["influx"] = load.model.n_reac - 1
        state["rate"] = float(load.model.k[state["influx"]]) * (1.0 + 4.0 * np.random.default_rng(seed).uniform())
    return state


def run(state):
    kind = state["kind"]
    if kind == "batch":
        for sim, counts in zip(state["sims"], state["counts"]):
            sim.set_counts(counts)
        state["batch"].run([sim.time + state["length"] for sim in state["sims"]])
        return [sim.get_counts(out) for sim, out in zip(state["sims"], state["results"])]
    if kind == "served":
        server = state["server"]
        ids = [server.submit(proto, seed, counts, t) for proto, seed, counts, t in state["jobs"]]
        while server.step()[0] > 0:
            pass
        return [server.take_result(job) for job in ids]
    sim = state["sim"]
    if kind == "noalloc":
        state["work"].copy_(state["initial"])
        capi.steps_run_noalloc(sim._sim, state["work"].data_ptr(), sim.time + state["length"])
        return state["work"]
    sim.set_counts(state["counts"])
    if kind == "record":
        sim.set_reac_rate(state["influx"], state["rate"])
        n = sim.run_record(sim.time + state["length"], state["every"], state["species"], state["tets"],
                           state["records"].data_ptr(), state["records"].shape[0])
        return {"recordings": n, "records": state["records"], "counts": sim.get_counts(state["result"])}
    sim.run(sim.time + state["length"])
    return sim.get_counts(state["result"])


# ---------------------------------------------------------------- what a pass cannot do without

def _update_bytes(load):
    """Bytes of one tet in one window: every count in and out (4 bytes each),
    four neighbours, four leave probabilities, the volume factor, and the
    active-reaction word where reactions are limited to a region."""
    return 8 * load.model.n_species + 36 + (4 if load.masks else 0)


def work(case):
    if case["kind"] == "batch":
        loads = [_box(17, nx, 17, 17, 1.0) for nx in _box_lengths(case)]
        parts = [(loads[j % case["meshes"]], case["windows"]) for j in range(case["members"])]
    elif case["kind"] == "served":
        parts = [(_job_load(family, size), windows) for family, size, windows in _jobs(case)]
    else:
        parts = [(_load(case), case["windows"])]
    return {"bytes": sum(load.nt * math.ceil(windows) * _update_bytes(load) for load, windows in parts), "flops": 0}


def exact(case, seed):
    """Outputs are whole numbers, the same on every side: nothing to compare in 64 bits."""
    return None
