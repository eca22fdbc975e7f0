"""Measured cases of the shower transport: whole calls through the public binding.

A case is one of

* ``transport``: submit one or more requests of primaries, transport them until the last
  track dies, and take every request's per-event deposits back to the host;
* ``image``: a ray-traced image of a calorimeter into device memory;
* ``tables``: the allocation-free build of the physics tables and production thresholds.

Geometries, materials, fields and primary recipes are those of
``paper_2209_15445_gb300.workloads``. Contexts (arena, tables, captured graphs) are what a
program keeps, so they belong to the state; the requests are made from the seed.
"""
import math

import numpy as np
import torch

from paper_2209_15445_gb300 import adept as A
from paper_2209_15445_gb300 import workloads as W

GEOMETRIES = {"slab": W.slab_calorimeter, "pbwo4": W.pbwo4_calorimeter, "barrel": W.barrel_calorimeter}
ELEMENTS = {"Pb": W.PB, "lAr": W.LAR, "Si": W.SI, "Fe": W.FE}

# tracked steps per MeV of primary energy, rounded (what a shower of these geometries takes)
STEPS_PER_MEV = {"slab": 5.6, "pbwo4": 5.0, "barrel": 4.3}
MSC_STEPS = 6.0  # multiple scattering limits the steps: so many times more of them


def _transport(name, geometry, beam, n, E, precision=1, field=0.0, physics=0, chord=0, requests=1,
               device=False, fused=0, generations=0):
    return {"name": name, "kind": "transport", "geometry": geometry, "beam": beam, "n": n, "E": E,
            "precision": precision, "field": field, "physics": physics, "chord": chord, "requests": requests,
            "device": device, "fused": fused, "generations": generations}


def _image(name, geometry, view, nx, ny, precision):
    return {"name": name, "kind": "image", "geometry": geometry, "view": view, "nx": nx, "ny": ny,
            "precision": precision}


def _tables(name, materials, cut_mm):
    return {"name": name, "kind": "tables", "materials": materials, "cut_mm": cut_mm}


def listed():
    return [
        # one particle handed over by a host simulation: nothing to batch, latency of the call
        _transport("one_shower", "slab", "electrons", 1, 1e4),
        # the plain FP64 form on its small validation sample: 100 electrons of 1 GeV
        _transport("fp64_100x1GeV", "slab", "electrons", 100, 1e3, precision=0),
        # a validation run of the plain FP64 form that fills the GPU
        _transport("fp64_300x10GeV", "slab", "electrons", 300, 1e4, precision=0),
        # fast simulation of a detector region in the lead-tungstate calorimeter: an odd batch
        _transport("pbwo4_997", "pbwo4", "electrons", 997, 1e4),
        # the benchmark's batch of 10,000 showers, primaries already in device memory
        _transport("batch_10000", "slab", "electrons", 10000, 1e4, device=True),
        # uneven primaries (species, 0.1 to 100 GeV) in a field along the beam
        _transport("mixed_1T", "slab", "mixed", 12000, 0.0, field=1.0),
        # a collider barrel in its solenoid field: many requests, the largest call
        _transport("barrel_3.8T", "barrel", "barrel", 40000, 0.0, field=3.8, requests=40),
        # the same barrel with the chord propagator of the field, capped at 100 iterations; about
        # one primary in 300 leaves a track that loops until the step cap (10,000 steps here) ends it
        _transport("barrel_chords", "barrel", "barrel", 1500, 0.0, field=3.8, chord=100),
        # the optional physics: multiple scattering and loss fluctuations
        _transport("slab_msc_fluct", "slab", "electrons", 501, 1e4, physics=3),
        # serving: a round of requests of very different sizes, one event each, one kernel per generation
        _transport("serving_round", "barrel", "serving", 16, 0.0, field=3.8, requests=16, fused=1, generations=8),
        # a ray-traced check of the barrel with the split form's FP32 distances
        _image("image_barrel", "barrel", "side", 2048, 2047, 1),
        # physics tables and thresholds of one calorimeter, as at every new cut
        _tables("tables_Pb_lAr", "Pb,lAr", 0.7),
    ]


def _log(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def draw(rng):
    kind = rng.choice(["electrons", "electrons", "fp64", "mixed", "barrel", "chords", "physics", "serving", "image",
                       "tables"])
    if kind in ("electrons", "fp64", "physics"):
        E = round(_log(rng, 200.0, 5e4), 1)
        split = kind != "fp64"
        most = {"electrons": 1.2e8, "fp64": 6e6, "physics": 8e6}[kind]  # MeV of one pass
        n = max(1, int(_log(rng, 1.0, min(2e4, most / E))))
        c = _transport("", rng.choice(["slab", "pbwo4"]), "electrons", n, E, precision=1 if split else 0,
                       physics=rng.choice([1, 3]) if kind == "physics" else 0, device=rng.random() < 0.4)
    elif kind == "mixed":
        c = _transport("", rng.choice(["slab", "pbwo4"]), "mixed", int(_log(rng, 10.0, 1.2e4)), 0.0,
                       field=rng.choice([0.0, 0.5, 1.0, 2.0]))
    elif kind == "barrel":
        n = int(_log(rng, 50.0, 3e4))
        c = _transport("", "barrel", "barrel", n, 0.0, field=rng.choice([1.0, 2.0, 3.8]),
                       requests=max(1, min(n, int(_log(rng, 1.0, 40.0)))))
    elif kind == "chords":
        c = _transport("", "barrel", "barrel", int(_log(rng, 20.0, 1000.0)), 0.0, field=rng.choice([1.0, 2.0, 3.8]),
                       chord=rng.choice([10, 30, 100]))
    elif kind == "serving":
        n = rng.randint(2, 20)
        c = _transport("", "barrel", "serving", n, 0.0, field=3.8, requests=n, fused=rng.choice([0, 1]),
                       generations=rng.choice([8, 16, 32]))
    elif kind == "image":
        c = _image("", *rng.choice([("slab", "oblique"), ("slab", "front"), ("barrel", "side"), ("barrel", "end")]),
                   int(_log(rng, 300.0, 2400.0)), int(_log(rng, 300.0, 2400.0)), rng.choice([0, 1]))
    else:
        names = rng.sample(sorted(ELEMENTS), rng.randint(1, 4))
        c = _tables("", ",".join(names), round(_log(rng, 0.1, 3.0), 3))
    del c["name"]
    return c


# ---------------------------------------------------------------- inputs
def _energy(case):
    """mean primary energy of the case, MeV (all primaries together)"""
    per = {"electrons": case["E"], "mixed": (1e5 - 100.0) / math.log(1000.0), "barrel": 4.9e4 / math.log(50.0),
           # 1/E uniform between 1/10 MeV and 1/20 GeV; sizes log-uniform in 10 .. 10,000
           "serving": 10.0 * math.log(2000.0) * (1e4 - 10.0) / math.log(1000.0)}
    return case["n"] * per[case["beam"]]


def _primaries(case, seed):
    n, first = case["n"], (seed * 1000003) % (1 << 30)
    if case["beam"] == "electrons":
        parts = [W.electrons(n, case["E"], first_event=first)]
    elif case["beam"] == "mixed":
        parts = [W.mixed(n, seed=seed, first_event=first)]
    elif case["beam"] == "barrel":
        p = W.barrel_primaries(n, seed=seed, first_event=first)
        k = case["requests"]
        parts = [p.take(np.arange(i * n // k, (i + 1) * n // k)) for i in range(k)]
    else:  # one batch of tracks of one event for each producer
        # sizes spread over the logarithm of their range, the same for every seed
        parts = [W.serving_batch(int(10.0 * 1000.0 ** ((i + 0.5) / n)), seed=seed * 131 + i, event=first + i)
                 for i in range(n)]
    return parts


def _camera(view, seed):
    rng = np.random.default_rng(seed)
    a, b = rng.uniform(0.02, 0.12, 2)
    return {"oblique": [-600.0, 50.0, -300.0, 1.0, a, 0.6 + b, 0, 0, 1, 500.0, 700.0],
            "front": [0.0, 0.0, -50.0, a, b, 1.0, 0, 1, 0, 500.0, 500.0],
            "side": [-4000.0, 0.0, 0.0, 1.0, a, b, 0, 0, 1, 3800.0, 6500.0],
            "end": [0.0, 0.0, -5000.0, a, b, 1.0, 1, 0, 0, 3800.0, 3800.0]}[view]


def _materials(case):
    return [ELEMENTS[m] for m in case["materials"].split(",")]


def prepare(case, seed):
    if case["kind"] == "tables":
        mats = _materials(case)
        u = float(np.random.default_rng(seed).uniform(0.95, 1.05))
        return {"kind": "tables", "materials": mats, "cut": case["cut_mm"] * u,
                "tables": torch.empty((len(mats), 12, A.NNODE), dtype=torch.float64, device="cuda"),
                "cuts": torch.empty((len(mats), 2), dtype=torch.float64, device="cuda")}
    geom = GEOMETRIES[case["geometry"]]()
    if case["kind"] == "image":
        tr = A.Transport(geom, precision=case["precision"], field_T=0.0, arena_bytes=256 << 20, max_events=1024)
        nx, ny = case["nx"], case["ny"]
        return {"kind": "image", "tr": tr, "precision": case["precision"], "nx": nx, "ny": ny,
                "camera": np.array(_camera(case["view"], seed)),
                "image": torch.empty((ny, nx, 2), dtype=torch.float64, device="cuda")}
    parts = _primaries(case, seed)
    energy = float(sum(p.E.sum() for p in parts))
    opts = {}
    if case["physics"]:
        opts["physics"] = case["physics"]
    if case["chord"]:
        opts["field_max_iterations"] = case["chord"]
        opts["max_steps"] = 10000
    if case["fused"]:
        opts["fused"] = 1
    if case["generations"]:
        opts["graph_generations"] = case["generations"]
    arena = int(min(24e9, 2e9 + energy * (700.0 if case["physics"] else 130.0)))
    tr = A.Transport(geom, precision=case["precision"], field_T=case["field"], arena_bytes=arena, max_events=65536,
                     tracks_per_MeV=0.1, **opts)
    tracks = [A.tracks_array(p) for p in parts]
    events = [len(np.unique(p.event)) for p in parts]
    return {"kind": "transport", "tr": tr, "events": events,
            "tracks": [torch.from_numpy(t.view(np.uint8).copy()).cuda() for t in tracks] if case["device"] else tracks,
            "sizes": [len(t) for t in tracks], "device": case["device"],
            "rows": [np.empty((n, tr.n_bins)) for n in events]}


# ---------------------------------------------------------------- one pass
def run(state):
    if state["kind"] == "tables":
        # the current stream: calls that overlap on the GPU would share the build's static scratch
        rc = A.adept_build_tables_noalloc(state["materials"], state["cut"], state["tables"].data_ptr(),
                                          state["cuts"].data_ptr(), torch.cuda.current_stream().cuda_stream)
        if rc != A.OK:
            raise A.AdeptError(rc, "table build")
        return {"tables": state["tables"], "cuts": state["cuts"]}
    tr = state["tr"]
    if state["kind"] == "image":
        tr.check(A.adept_raytrace_device(tr.h, state["precision"], state["camera"], state["nx"], state["ny"],
                                         state["image"].data_ptr()))
        return state["image"]
    if state["device"]:
        ids = [tr.submit_device(t, n) for t, n in zip(state["tracks"], state["sizes"])]
    else:
        ids = [tr.submit(t) for t in state["tracks"]]
    tr.transport()
    totals = []
    for rid, n, rows in zip(ids, state["events"], state["rows"]):
        _, meta = tr.result(rid, n, out=rows)
        totals.append((meta.deposited_MeV, meta.leaked_MeV, meta.killed_MeV))
    return {"deposits": state["rows"][0] if len(state["rows"]) == 1 else np.concatenate(state["rows"]),
            "totals": np.array(totals)}


# ---------------------------------------------------------------- what a pass cannot do without
def work(case):
    if case["kind"] == "tables":
        n = len(case["materials"].split(","))
        # 11 rows of closed forms of about 40 operations and three ranges of 8 panels a bin
        return {"bytes": n * (12 * 289 + 2) * 8.0, "flops": n * 289 * (11 + 3 * 17) * 40.0}
    if case["kind"] == "image":
        pixels = case["nx"] * case["ny"]
        crossings = {"oblique": 60.0, "front": 60.0, "side": 90.0, "end": 90.0}[case["view"]]
        return {"bytes": 16.0 * pixels, "flops": pixels * crossings * 25.0}
    geom = GEOMETRIES[case["geometry"]]()
    tracks = case["n"]
    if case["beam"] == "serving":
        tracks = sum(int(10.0 * 1000.0 ** ((i + 0.5) / case["n"])) for i in range(case["n"]))
    steps = _energy(case) * STEPS_PER_MEV[case["geometry"]] * (MSC_STEPS if case["physics"] else 1.0)
    # about 150 operations a step: four table entries, an interaction length, a boundary
    # distance, a move, the loss and a share of an interaction
    return {"bytes": 72.0 * tracks + 8.0 * case["n"] * geom.n_bins, "flops": steps * 150.0}


# ---------------------------------------------------------------- 64-bit values where there are any
def exact(case, seed):
    """The images have closed forms. A shower has none: its value is its random history."""
    if case["kind"] != "image":
        return None
    geom = GEOMETRIES[case["geometry"]]()
    cam = _camera(case["view"], seed)
    nx, ny = case["nx"], case["ny"]
    o, d, up = (np.array(cam[k:k + 3], float) for k in (0, 3, 6))
    d /= np.linalg.norm(d)
    right = np.cross(d, up)
    right /= np.linalg.norm(right)
    up = np.cross(right, d)
    f8 = dict(dtype=torch.float64, device="cuda")
    a = ((torch.arange(nx, **f8) + 0.5) / nx - 0.5) * cam[9]
    b = ((torch.arange(ny, **f8) + 0.5) / ny - 0.5) * cam[10]
    p = [o[k] + a[None, :] * right[k] + b[:, None] * up[k] for k in range(3)]
    big = 1e300

    def between(lo, hi, axis):  # path parameters where lo <= p + t d <= hi on one axis
        if d[axis] == 0.0:
            inside = (p[axis] >= lo) & (p[axis] <= hi)
            return torch.where(inside, -big, big), torch.where(inside, big, -big)
        t = [(v - p[axis]) / d[axis] for v in (lo, hi)]
        return torch.minimum(*t), torch.maximum(*t)

    density = [m.density for m in geom.materials]
    if geom.kind == 0:
        z = np.concatenate([[0.0], np.cumsum(np.tile(geom.sub_thickness, geom.n_layers))])
        t0, t1 = between(z[0], z[-1], 2)
        for axis in (0, 1):
            s0, s1 = between(-geom.half_xy, geom.half_xy, axis)
            t0, t1 = torch.maximum(t0, s0), torch.minimum(t1, s1)
        t0 = t0.clamp_min(0.0)
        mass, count = torch.zeros_like(t0), torch.zeros_like(t0)
        for v in range(len(z) - 1):
            s0, s1 = between(z[v], z[v + 1], 2)
            path = (torch.minimum(s1, t1) - torch.maximum(s0, t0)).clamp_min(0.0)
            mass += density[geom.sub_materials[v % geom.n_sub]] * 0.1 * path
            count += path > 0.0
        return torch.stack([mass, count], -1)
    thick = np.concatenate([[0.0], np.cumsum(geom.sub_thickness)])
    aa = d[0] * d[0] + d[1] * d[1]
    bb = p[0] * d[0] + p[1] * d[1]
    r2 = p[0] * p[0] + p[1] * p[1]

    def chord(radius):
        disc = bb * bb - aa * (r2 - radius * radius)
        s = torch.sqrt(disc.clamp_min(0.0))
        return torch.where(disc > 0, (-bb - s) / aa, big), torch.where(disc > 0, (-bb + s) / aa, -big)

    t0, t1 = chord(geom.layer_r[-1] + thick[-1])
    s0, s1 = between(-geom.half_z, geom.half_z, 2)
    t0, t1 = torch.maximum(t0, s0).clamp_min(0.0), torch.minimum(t1, s1)
    hit = t1 > t0
    mass, count = torch.zeros_like(t0), hit.to(torch.float64)
    for r in geom.layer_r:
        inner = None
        for v, radius in enumerate(r + thick):
            s0, s1 = chord(radius)
            path = (torch.minimum(s1, t1) - torch.maximum(s0, t0)).clamp_min(0.0)
            for s in (s0, s1):  # a crossing strictly inside the world enters another volume
                if not (r == geom.layer_r[-1] and v == len(thick) - 1):
                    count += (hit & (s > t0) & (s < t1)).to(torch.float64)
            if inner is not None:
                mass += density[geom.sub_materials[v - 1]] * 0.1 * (path - inner)
            inner = path
    return torch.stack([mass * hit, count], -1)
