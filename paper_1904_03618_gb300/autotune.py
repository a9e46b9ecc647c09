"""Launch-configuration autotuner for the fused step.

The fused kernel's launch configuration -- tile height, planes per CTA
(z chunk) and where a plane's reduced state waits between its pull and its
collision -- changes results by rounding only (the parity tests run every
configuration against the oracle), and the best choice depends on the
lattice shape, the storage type and, for batches, on the mix of box sizes.
`tune` times the candidate configurations on the live context with CUDA
events on its stream, among them what lbm_create picks (on small lattices
the box form), keeps the fastest, applies it, and records it in a JSON cache
keyed by device, storage, collision operator and lattice signature so that
later runs of the same shape skip the timing.

Timing advances the context's state (it runs real steps).  Tune before
initialising the run that matters, or accept the extra steps.
"""
from __future__ import annotations

import json
import os
import time

import torch

from . import lbm

# (tile_y, hold) shapes; z chunks are tried for each
SINGLE_SHAPES = [(8, 2), (8, 7), (8, 8), (16, 8), (16, 7), (8, 3), (8, 0), (16, 1), (16, 4)]
BATCH_SHAPES = [(12, 7), (8, 2), (15, 7), (15, 8), (8, 7), (8, 0), (16, 1)]
# z chunks: longer chunks pay fewer halo planes, and beyond about 48 planes
# the CTAs of neighbouring columns drift apart (their shared halo lines miss
# in L2); the timing decides
ZCHUNKS = [8, 12, 16, 24, 32, 48, 64]

DEFAULT_CACHE = os.path.join(os.path.expanduser("~"), ".cache", "paper_1904_03618_gb300",
                             "autotune.json")


# of the library's set of forms: entries timed among other forms do not apply
FORMS = 2


def signature(params_list, storage: int) -> str:
    """Cache key of a lattice (one params) or a batch (several)."""
    dev = torch.cuda.get_device_name()
    if len(params_list) == 1:
        p = params_list[0]
        shape = "%dx%dx%d/w%d%d%d" % (p.nx, p.ny, p.nz, p.wall[0], p.wall[1], p.wall[2])
    else:
        sizes = sorted((p.nx, p.ny, p.nz) for p in params_list)
        counts = {}
        for s in sizes:
            counts[s] = counts.get(s, 0) + 1
        shape = "batch:" + ",".join("%dx%dx%d*%d" % (k + (v,)) for k, v in sorted(counts.items()))
    return "%s|storage%d|%s|collision%d|forms%d" % (dev, storage, shape, params_list[0].collision,
                                                    FORMS)


def _load(path):
    try:
        with open(path) as fh:
            return json.load(fh)
    except (OSError, ValueError):
        return {}


def _store(path, table):
    os.makedirs(os.path.dirname(path), exist_ok=True)
    tmp = path + ".tmp%d" % os.getpid()
    with open(tmp, "w") as fh:
        json.dump(table, fh, indent=1, sort_keys=True)
    os.replace(tmp, path)


def _apply(ctx, tile_y, zchunk, hold, box):
    """The configuration, or with box > 0 the box form beside it."""
    lbm.lbm_set_fused_config(ctx, tile_y, zchunk, hold)
    if box:
        lbm.lbm_set_box(ctx, box)


def _time(ctx, stream, steps):
    e0 = torch.cuda.Event(enable_timing=True)
    e1 = torch.cuda.Event(enable_timing=True)
    warmup = 4  # captures the graph that the timed steps replay
    if lbm.lbm_get_box(ctx):
        warmup, steps = 20, max(steps, 32)  # 16 steps to a graph
    lbm.lbm_step(ctx, warmup)
    e0.record(stream)
    lbm.lbm_step(ctx, steps)
    e1.record(stream)
    stream.synchronize()
    return e0.elapsed_time(e1) / steps


def tune(ctx, params_list, stream, steps=8, cache_path=DEFAULT_CACHE, use_cache=True,
         candidates=None):
    """Chooses and applies the fastest fused configuration for `ctx` (a
    Lattice's or Batch's context; every case must be initialised).  Returns
    (tile_y, zchunk, hold, ms_per_step, source) with source "cache" or
    "timed"; whether the box form steps beside it, lbm_get_box tells."""
    params_list = list(params_list)
    storage = int(params_list[0].storage)
    key = signature(params_list, storage)
    table = _load(cache_path) if (use_cache and cache_path) else {}
    if use_cache and key in table:
        t = table[key]
        try:
            _apply(ctx, t["tile_y"], t["zchunk"], t["hold"], t["box"])
            return t["tile_y"], t["zchunk"], t["hold"], t["ms"], "cache"
        except (KeyError, lbm.LbmError):
            pass  # not of this context after all: time it
    if candidates is None:
        shapes = BATCH_SHAPES if len(params_list) > 1 else SINGLE_SHAPES
        nz = max(p.nz for p in params_list)
        candidates = [(ty, zc, hold) for ty, hold in shapes for zc in ZCHUNKS if zc <= max(nz, 8)]
        if len(params_list) == 1:  # what lbm_create picks, whatever the context runs now
            sms = torch.cuda.get_device_properties(torch.cuda.current_device()).multi_processor_count
            p = params_list[0]
            candidates.insert(0, lbm.lbm_default_fused_config(p, sms) + (lbm.lbm_default_box(p),))
    best = None
    for ty, zc, hold, box in (tuple(c) + (0,) * (4 - len(c)) for c in candidates):
        try:
            _apply(ctx, ty, zc, hold, box)
        except lbm.LbmError:
            continue
        ms = _time(ctx, stream, steps)
        if best is None or ms < best[4]:
            best = (ty, zc, hold, box, ms)
    if best is None:
        raise RuntimeError("autotune: no valid configuration")
    ty, zc, hold, box, ms = best
    _apply(ctx, ty, zc, hold, box)
    if cache_path:
        table = _load(cache_path)
        table[key] = {"tile_y": ty, "zchunk": zc, "hold": hold, "box": box, "ms": ms,
                      "when": time.strftime("%Y-%m-%dT%H:%M:%S")}
        _store(cache_path, table)
    return ty, zc, hold, ms, "timed"
