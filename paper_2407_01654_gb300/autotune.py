"""Autotuner for the per-simulation launch schedule of the coupled step.

For one lattice shape (nx, ny, walls, storage precision), potential scheme and kind of count
(the stopping rule's or a fixed one) it times every candidate schedule of the potential loop -- the streaming kernel (one launch per sub-iteration in a
graph WHILE node), the resident on-chip loop and the on-chip loops with two and three
sub-iterations per exchange, each with every tile height of 64-wide tiles (`tile_rows`;
0 = the built-in choice of about 2048 nodes per tile) -- on a short run with
a set number of sub-iterations, and returns the fastest as parameter overrides.  All
candidates compute the same bits at a fixed sub-iteration count (the tests check this), so
tuning changes speed only.  Results are cached per device and shape_key, for the library whose
kernels were timed, in a JSON file ($EHD_AUTOTUNE_CACHE, else
~/.cache/paper_2407_01654_gb300/autotune.json).

    from paper_2407_01654_gb300 import autotune
    params.update(autotune.tune(params))
"""
from __future__ import annotations

import hashlib
import json
import os
import time

import numpy as np

TILE_ROWS = (0, 8, 16, 24, 32, 40, 48, 56, 64)
LOOP_STREAM, LOOP_RESIDENT, LOOP_RESIDENT2, LOOP_RESIDENT3 = 1, 2, 3, 4


def candidates(params):
    """Parameter overrides to try: the streaming loop, then the resident loop at each
    tile height (the library refuses heights whose tiles do not fit on chip)."""
    ny = params["ny"]
    rows = [r for r in TILE_ROWS[1:] if r <= ny]
    taller = [r for r in TILE_ROWS[1:] if r > ny]
    if taller:
        rows.append(taller[0])  # one row of tiles; taller heights only add idle threads
    out = [{"poisson_loop": LOOP_STREAM, "tile_rows": 0},
           {"poisson_loop": LOOP_RESIDENT, "tile_rows": 0}]
    out += [{"poisson_loop": LOOP_RESIDENT, "tile_rows": r} for r in rows]
    # two sub-iterations per exchange: tiles of 24 rows or more; three: 48 or more
    out += [{"poisson_loop": LOOP_RESIDENT2, "tile_rows": 0}]
    out += [{"poisson_loop": LOOP_RESIDENT2, "tile_rows": r} for r in rows if r >= 24]
    out += [{"poisson_loop": LOOP_RESIDENT3, "tile_rows": 0}]
    out += [{"poisson_loop": LOOP_RESIDENT3, "tile_rows": r} for r in rows if r >= 48]
    return out


def shape_key(params, device_name):
    """What a schedule is tuned for.  The conventional potential scheme has a key of its own:
    the loops are other kernels, and one of them (three sub-iterations per exchange) does not
    exist for it.  So has a fixed count, which runs another kernel than the stopping rule."""
    return (f"{device_name}|{params['nx']}x{params['ny']}|walls{params['walls_y']}"
            f"|prec{params['precision']}" + ("|conv" if params.get("potential_scheme") else "")
            + ("|fixed" if params.get("poisson_fixed_iter") else ""))


def library_id():
    """Identifies the kernels that timings belong to: a hash of the library's sources and build
    flags.  Cached schedules of another library are not used, since they say nothing about
    this one."""
    from . import build
    paths = [os.path.abspath(build.__file__)]
    for d in (build.CSRC, os.path.join(build.ROOT, "include")):
        try:
            paths += [os.path.join(d, n) for n in sorted(os.listdir(d))
                      if n.endswith((".cu", ".cuh", ".h"))]
        except OSError:
            pass  # a library installed without its sources
    h = hashlib.sha256()
    for p in paths:
        with open(p, "rb") as fh:
            h.update(os.path.basename(p).encode() + b"\0" + fh.read() + b"\0")
    return h.hexdigest()[:16]


def cache_path():
    p = os.environ.get("EHD_AUTOTUNE_CACHE")
    if p:
        return p
    return os.path.join(os.path.expanduser("~"), ".cache", "paper_2407_01654_gb300",
                        "autotune.json")


def load_cache(path):
    try:
        with open(path) as fh:
            return json.load(fh)
    except (OSError, ValueError):
        return {}


def cached(path, key):
    """The cached entry of this key if this library's kernels were timed for it, else None."""
    hit = load_cache(path).get(key)
    return hit if hit and hit.get("library") == library_id() else None


def store_cache(path, key, entry):
    d = load_cache(path)
    d[key] = dict(entry, library=library_id())
    try:
        os.makedirs(os.path.dirname(path), exist_ok=True)
        tmp = path + ".tmp"
        with open(tmp, "w") as fh:
            json.dump(d, fh, indent=1, sort_keys=True)
        os.replace(tmp, path)
    except OSError:
        pass  # a read-only home only costs a re-tune


def pick(timings):
    """The fastest candidate; ties go to the earlier one.  timings: [(overrides, seconds
    or None when the candidate could not run)]."""
    best = None
    for ov, t in timings:
        if t is None or not np.isfinite(t):
            continue
        if best is None or t < best[1]:
            best = (ov, t)
    if best is None:
        raise RuntimeError("no candidate schedule could run")
    return best


def time_candidate(params, fields, overrides, steps, fixed_iter):
    """Seconds per step of `steps` coupled steps with `fixed_iter` sub-iterations each,
    after two warm-up steps; None if the library rejects the schedule.  Parameters under the
    stopping rule are timed with the rule's kernels: a smallest count equal to the largest, and
    a tolerance (within FP32's range when squared) that no solve of that length reaches."""
    from . import ehd
    p = dict(params)
    p.update(overrides)
    if params.get("poisson_fixed_iter"):
        p["poisson_fixed_iter"] = fixed_iter
    else:
        p.update(poisson_min_iter=fixed_iter, poisson_max_iter=fixed_iter, poisson_tol=1e-12)
    try:
        sim = ehd.Sim(p)
    except ehd.EhdError:
        return None
    try:
        if overrides["poisson_loop"] != sim.loop_kind():
            return None
        sim.set_fields(fields["phi"], fields["q"], fields["ux"], fields["uy"])
        sim.step(2, stats=False)
        sim.read_stats()  # synchronises
        t0 = time.perf_counter()
        sim.step(steps, stats=False)
        sim.read_stats()
        return (time.perf_counter() - t0) / steps
    finally:
        sim.close()


def tune(params, fields=None, steps=20, fixed_iter=32, use_cache=True, timer=None,
         device_name=None):
    """Parameter overrides ({"poisson_loop", "tile_rows"}) of the fastest schedule for this
    lattice shape.  `fields`: initial fields to time with (default: a flat interface at
    mid-height); `timer(params, fields, overrides, steps, fixed_iter)` replaces the GPU
    timing (tests)."""
    if device_name is None:
        device_name = _device_name()
    key = shape_key(params, device_name)
    path = cache_path()
    if use_cache:
        hit = cached(path, key)
        if hit:
            return dict(hit["overrides"])
    if fields is None:
        fields = _default_fields(params)
    timer = timer or time_candidate
    timings = [(ov, timer(params, fields, ov, steps, fixed_iter)) for ov in candidates(params)]
    ov, t = pick(timings)
    if use_cache:
        store_cache(path, key, {"overrides": ov, "seconds_per_step": t,
                                "timings": [[o, s] for o, s in timings]})
    return dict(ov)


def _device_name():
    try:
        import torch
        return torch.cuda.get_device_name(0).replace(" ", "_")
    except Exception:
        return "unknown"


def _default_fields(params):
    ny, nx = params["ny"], params["nx"]
    y = np.arange(ny, dtype=float)[:, None] + np.zeros((1, nx))
    phi = 0.5 + 0.5 * np.tanh(2.0 * (ny / 2.0 - y) / params["width"])
    z = np.zeros((ny, nx))
    return {"phi": phi, "q": z, "ux": z, "uy": z}


# ---------------------------------------------------------------------------------------
# Batches: one schedule for all slots (tile height and steps per captured graph)
# ---------------------------------------------------------------------------------------

BATCH_ROWS = (16, 32, 64)
BATCH_STEPS_PER_GRAPH = (8, 16, 32)


def batch_candidates():
    return [{"tile_rows": r, "steps_per_graph": g} for r in BATCH_ROWS
            for g in BATCH_STEPS_PER_GRAPH]


def time_batch_candidate(requests, schedule, steps, budget):
    """Node updates per second of a batch holding as many of `requests` (params, fields)
    as it admits under `schedule`, over `steps` steps after a warm-up; None if none fit."""
    from . import ehd
    b = ehd.Batch(budget, max_slots=len(requests), steady_tol=1e-30, step_cap=1 << 40)
    try:
        b.set_schedule(**schedule)
        nodes = 0
        for i, (p, f) in enumerate(requests):
            if b.admit(p, f, i) is not None:
                nodes += p["nx"] * p["ny"]
        if nodes == 0:
            return None
        b.run(2)
        t0 = time.perf_counter()
        b.run(steps)
        return nodes * steps / (time.perf_counter() - t0)
    finally:
        b.close()


def tune_batch(requests, steps=64, budget=2 << 30, use_cache=True, timer=None,
               device_name=None):
    """Batch schedule ({"tile_rows", "steps_per_graph"}) with the most node updates per
    second on a sample of requests [(params, fields)]; cached per device and mix of
    lattice shapes.  `timer(requests, schedule, steps, budget)` replaces the GPU timing."""
    if device_name is None:
        device_name = _device_name()
    shapes = sorted(f"{p['nx']}x{p['ny']}" for p, _ in requests)
    key = f"{device_name}|batch|{','.join(shapes)}"
    path = cache_path()
    if use_cache:
        hit = cached(path, key)
        if hit:
            return dict(hit["overrides"])
    timer = timer or time_batch_candidate
    rates = [(s, timer(requests, s, steps, budget)) for s in batch_candidates()]
    # the fastest is the one with the smallest inverse rate
    best, inv = pick([(s, None if r is None else 1.0 / r) for s, r in rates])
    if use_cache:
        store_cache(path, key, {"overrides": best, "node_updates_per_s": 1.0 / inv,
                                "rates": [[s, r] for s, r in rates]})
    return dict(best)
