"""Autotuner for the line-solver launch parameters of one grid shape.

Knobs (see ``adi_wave_tuning`` in include/adiwave.h): systems (rows) per CTA
of the x sweep, unknowns per thread in each sweep, strip width of the y sweep,
threads per CTA, the interface solver (warp-shuffle block CR + PCR, or
shared-memory CR handing `pcr_size` equations to warp PCR -- the CR-to-PCR
switch level) and graph replay.

The knobs are those of the separate sweeps.  A step that is one launch
(``AdiWave.plan()``: form other than "sweeps") has none, and setting any of them
would take it off that path: there the answer is the empty tuning, without a
search, unless the runs keep checkpoints and so take the sweeps.

Each candidate runs a few steps of a problem of the requested shape with
per-kernel CUDA events on the launching stream, at the handle's own tau and
bound of m (which decide where the elimination is in FP64; beyond that the
sweeps do the same work for any coefficient), keeping one checkpoint so that
the sweeps are what is timed.  The x-sweep and y-sweep knobs act on
different kernels: for each setting of the shared knobs (solver, CR-to-PCR
switch) the x candidates are timed with the y sweep on automatic, then the
y candidates with the best x.  The planner's automatic choice is timed
first and kept unless a searched tuning is faster (an empty tuning dict
means "automatic").  Results are cached per (device, nx, ny, precision) and
form of the step in a JSON file (``$ADIWAVE_TUNE_CACHE`` or
``~/.cache/adiwave/tuning.json``); entries of other versions of this search,
which may hold knobs for a step that has become one launch, are left alone.
"""
from __future__ import annotations

import itertools
import json
import os
from typing import Dict

X_KNOBS = ("chunk_x", "rows_per_cta", "cta_threads", "x_stage", "x_cluster")
Y_KNOBS = ("chunk_y", "cols_per_cta", "cta_threads_y", "y_stage")
SHARED_KNOBS = ("solver", "pcr_size")


def cache_path() -> str:
    return os.environ.get("ADIWAVE_TUNE_CACHE",
                          os.path.join(os.path.expanduser("~"), ".cache", "adiwave", "tuning.json"))


VERSION = 2


def _key(device_name: str, nx: int, ny: int, fp64: str, form: str = "") -> str:
    """form: what _form() says; without it the key of version 1."""
    key = "%s|%dx%d|%s" % (device_name, nx, ny, fp64)
    return "%s|v%d|%s" % (key, VERSION, form) if form else key


def _form(plan: Dict, ckpt_every: int) -> str:
    """What a handle's steps are made of: "one launch", or the sweeps and the
    precision of their eliminations."""
    if plan["form"] != "sweeps" and not ckpt_every:
        return "one launch"
    return "sweeps fp%d fp%d" % tuple(64 if plan[d] else 32 for d in ("fp64_x", "fp64_y"))


def _load_cache() -> Dict:
    try:
        with open(cache_path()) as f:
            return json.load(f)
    except (OSError, ValueError):
        return {}


def _store_cache(data: Dict) -> None:
    p = cache_path()
    os.makedirs(os.path.dirname(p), exist_ok=True)
    tmp = p + ".tmp.%d" % os.getpid()
    with open(tmp, "w") as f:
        json.dump(data, f, indent=1, sort_keys=True)
    os.replace(tmp, p)


def candidates(nx: int, ny: int):
    """(shared settings, x candidates, y candidates) for a grid shape."""
    shared = [dict(solver=1, pcr_size=0), dict(solver=2, pcr_size=8), dict(solver=2, pcr_size=32)]
    # stage 3 = the TMA-pipelined persistent sweeps, 2 = direct loads (x) or
    # L2 prefetch (y), 1 = shared-memory staging, 4 = (y only) persistent CTAs
    # whose column segments meet through global memory, 5 = (x only) the band
    # form, each row over a cluster of x_cluster CTAs
    xs = [dict(chunk_x=k, rows_per_cta=0, cta_threads=t, x_stage=s, x_cluster=0)
          for k, t, s in itertools.product((8, 16, 32), (256, 512, 1024), (3, 2))]
    xs += [dict(chunk_x=k, rows_per_cta=0, cta_threads=0, x_stage=5, x_cluster=c)
           for k, c in itertools.product((32, 16), (2, 4))]
    ys = [dict(chunk_y=k, cols_per_cta=w, cta_threads_y=t, y_stage=s)
          for k, w, t, s in itertools.product((8, 16, 32), (8, 16), (256, 512, 1024), (4, 3, 1, 2))]
    return shared, xs, ys


def search(measure, shared, xs, ys):
    """(total ms, tuning, x_ms, y_ms) of the best setting, or None.

    measure(cfg) returns (x_ms, y_ms) or None when the shape rejects cfg.
    The planner's own choice (the empty tuning, all knobs automatic) is the
    reference: a searched tuning replaces it only when it is faster.  For
    each shared setting the x knobs are chosen by the x time with the y
    sweep on automatic, then the y knobs by the y time with that x."""
    ref = measure({})
    best = (ref[0] + ref[1], {}, ref[0], ref[1]) if ref else None
    for sh in shared:
        bx = None
        for xc in xs:
            cfg = dict(sh)
            cfg.update(xc)
            r = measure(cfg)
            if r and (bx is None or r[0] < bx[0]):
                bx = (r[0], xc)
        if bx is None:
            continue
        by = None
        for yc in ys:
            cfg = dict(sh)
            cfg.update(bx[1])
            cfg.update(yc)
            r = measure(cfg)
            if r and (by is None or r[1] < by[0]):
                by = (r[1], yc)
        if by is None:
            continue
        tot = bx[0] + by[0]
        if best is None or tot < best[0]:
            t = dict(sh)
            t.update(bx[1])
            t.update(by[1])
            best = (tot, t, bx[0], by[0])
    return best


def tune(nx: int, ny: int, fp64: str = "auto", steps: int = 3, warmup: int = 1,
         use_cache: bool = True, verbose: bool = False, sim=None) -> Dict:
    """Best tuning for an nx x ny grid: {'tuning': {...}, 'x_ms': .., 'y_ms': ..}.

    For the steps of the handle ``sim`` if one is given, else for runs without
    checkpoints at tau = 0.5 h / max c.  x_ms and y_ms are times of the
    sweeps; for a step of one launch 'step_ms' is its time and they are those
    of the sweeps that runs with checkpoints take.
    """
    import torch

    from . import api

    dev = torch.device("cuda", torch.cuda.current_device())
    name = torch.cuda.get_device_name(dev)
    h = min(1.0 / (nx + 1), 1.0 / (ny + 1))
    dt, lx, ly, m_max, ckpt = 0.5 * h, 1.0, 1.0, 1.0, 0
    if sim is not None:
        m_max, ckpt = sim.plan()["m_max"], sim.ckpt_every
        dt, lx, ly = sim.dt, sim.lx, sim.ly
    m = torch.full((ny, nx), m_max, dtype=torch.float32, device=dev)
    t = api.AdiWave(m, torch.zeros_like(m), dt, lx=lx, ly=ly, fp64=fp64)
    form = _form(t.plan(), ckpt)
    key = _key(name, nx, ny, fp64, form)
    cache = _load_cache() if use_cache else {}
    if key in cache:
        t.close()
        return cache[key]

    def timed():
        t.run(warmup)
        t.profile(True)
        t.profile_read()
        t.run(steps)
        ms, cnt = t.profile_read()
        t.profile(False)
        return [a / max(c, 1) for a, c in zip(ms, cnt)]

    def measure(cfg):
        """(x_ms, y_ms) of one tuning, or None when the shape rejects it."""
        try:
            t.set_tuning(**cfg)
        except api.AdiError:
            return None
        r = tuple(timed()[:2])
        if verbose:
            print(json.dumps({"cfg": cfg, "x_ms": r[0], "y_ms": r[1]}))
        return r

    out = {}
    if form == "one launch":
        out["step_ms"] = timed()[2]
    t.set_checkpointing(max(steps, warmup))  # the sweeps, whatever the plan
    if form == "one launch":
        best = (0.0, {}) + measure({})
    else:
        best = search(measure, *candidates(nx, ny))
    t.sync_status()
    t.close()
    if best is None:
        raise RuntimeError("no tuning candidate is valid for %dx%d" % (nx, ny))
    out.update(tuning=best[1], x_ms=best[2], y_ms=best[3])
    if use_cache:
        cache = _load_cache()
        cache[key] = out
        _store_cache(cache)
    return out


def apply(sim, fp64: str = "auto", **kw) -> Dict:
    """Tune for sim's steps (cached) and set the result on the handle."""
    sim.set_tuning()  # the plan to look at is the automatic one
    if _form(sim.plan(), sim.ckpt_every) == "one launch":
        return {"tuning": {}}
    res = tune(sim.nx, sim.ny, fp64=fp64, sim=sim, **kw)
    sim.set_tuning(**res["tuning"])
    return res
