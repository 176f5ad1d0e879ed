"""Autotuner for the rasteriser's launch shape.

Picks the tile shape (8x8, 16x16, 32x8) by timing the projection, binning,
forward, loss and backward of one mapping iteration on the caller's own map and
views with CUDA events (Adam is independent of the choice and is left out, so
the map is not modified).  These tiles are whole 8x8 blocks, whose render kernels
take no notice of the staging batch and the pixels per thread: those come back
as the defaults, and the backward's pixels per thread as what a deterministic
plan of the tile asks for.
The choice is cached in a JSON file keyed by GPU name, view sizes and a
power-of-two bucket of the map size.

The tile shape changes which pixels a Gaussian may reach (its 3-sigma rect is
counted in whole tiles), so it changes the image slightly.  Every tile shape is
checked against the FP64 oracle by the test-suite.
"""
from __future__ import annotations

import json
import math
import os

import torch

from . import mapping

TILES = ((8, 8), (16, 16), (32, 8))
SMEM_BATCH = 128  # the rasteriser's default
REPEATS = 4  # timed iterations per tile, in units of `iters`


def cache_path():
    return os.environ.get("GS_AUTOTUNE_CACHE",
                          os.path.join(os.path.expanduser("~"), ".cache", "paper_2409_13055_gb300",
                                       "autotune.json"))


def cache_key(views, n, tight_rect=True):
    name = torch.cuda.get_device_name()
    sizes = ",".join(f"{v['width']}x{v['height']}x{v.get('channels', 3)}" for v in views)
    rects = "tight" if tight_rect else "square"
    return f"{name}|{sizes}|n2^{max(0, int(math.log2(max(1, n))))}|{rects}"


def _shape(tile):
    return dict(smem_batch=SMEM_BATCH, pixels_per_thread=1, smem_batch_bwd=SMEM_BATCH,
                pixels_per_thread_bwd=tile[0] * tile[1] // 32)


def _time_tile(views, gmap, targets_packed, lam, tile, iters, tight_rect=True):
    """Mean (total, forward, backward) milliseconds of project + bin + forward +
    loss + pixel adjoint + projection adjoint with one tile shape."""
    rast = mapping.fit_instance_capacity(views, gmap, tile=tile, tight_rect=tight_rect,
                                         **_shape(tile))
    m, g = gmap.gs_map(), gmap.gs_map_grad()
    ev = [torch.cuda.Event(enable_timing=True) for _ in range(5)]

    def once(record):
        if record:
            ev[0].record()
        rast.project(m)
        rast.bin_sort(gmap.n)
        if record:
            ev[1].record()
        rast.render_fwd()
        if record:
            ev[2].record()
        rast.loss_l1_ssim(targets_packed, lam)
        if record:
            ev[3].record()
        rast.render_bwd(m, g)
        if record:
            ev[4].record()

    for _ in range(2):
        once(False)
    tot = fwd = bwd = 0.0
    for _ in range(iters):
        once(True)
        torch.cuda.synchronize()
        tot += ev[0].elapsed_time(ev[4])
        fwd += ev[1].elapsed_time(ev[2])
        bwd += ev[3].elapsed_time(ev[4])
    return tot / iters, fwd / iters, bwd / iters


def autotune(views, gmap: mapping.GaussianMap, targets_packed, lam, iters=5, use_cache=True,
             verbose=False, tight_rect=True):
    """Returns dict(tile=(w, h), smem_batch, pixels_per_thread, smem_batch_bwd,
    pixels_per_thread_bwd, ms, timings=[...])."""
    key = cache_key(views, gmap.n, tight_rect)
    path = cache_path()
    cache = {}
    fields = ("smem_batch", "pixels_per_thread", "smem_batch_bwd", "pixels_per_thread_bwd")
    if use_cache and os.path.exists(path):
        try:
            with open(path) as f:
                cache = json.load(f)
        except (OSError, ValueError):
            cache = {}
        if key in cache:
            c = cache[key]
            return dict(tile=tuple(c["tile"]), ms=c["ms"], timings=[], cached=True,
                        **{k: c[k] for k in fields})
    timings = []
    for tile in TILES:
        t = _time_tile(views, gmap, targets_packed, lam, tile, REPEATS * iters, tight_rect)
        timings.append(dict(tile=tile, smem_batch=SMEM_BATCH, pixels_per_thread=1, ms=t[0],
                            fwd_ms=t[1], bwd_ms=t[2]))
        if verbose:
            print(f"autotune {tile}: total {t[0]:.3f} fwd {t[1]:.3f} bwd {t[2]:.3f} ms")
    best = min(timings, key=lambda r: r["ms"])
    tile = best["tile"]
    out = dict(tile=tile, ms=best["ms"], timings=timings, cached=False, **_shape(tile))
    if use_cache:
        cache[key] = dict(tile=list(tile), ms=out["ms"], **{k: out[k] for k in fields})
        try:
            os.makedirs(os.path.dirname(path), exist_ok=True)
            tmp = path + f".tmp{os.getpid()}"
            with open(tmp, "w") as fh:
                json.dump(cache, fh, indent=1)
            os.replace(tmp, path)
        except OSError:
            pass
    return out
