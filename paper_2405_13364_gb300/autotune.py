"""Autotuner for the rasteriser's launch parameters.

Tunable here: the per-pixel sorter capacity K (the paper's depth-filter size, Sec. 2
"Sample blending"), the rasteriser's set-up (per warp, or shared by a CTA, Sec. 2,
Stage 3), the bin size of the binning stage (16, 32 or 64 pixels; Sec. 2, Stage 2
uses 32 and Sec. 4 proposes 64 and 16 for sparse and dense regions), the number of
persistent rasteriser CTAs per SM, and for flat-colour scenes whether the sorter carries
colours. Every candidate gives the same coverage and the same exact fragment order; K only
moves pixels between the sorter and the exact overflow path, whose composite sums in a
different order, so colours agree to fp32 rounding (the tuner checks 1e-5, the accuracy
bar) rather than bit for bit. The work item is an 8x4 half-block or an 8x8 block per
warp, or (shared set-up) a 32x8 strip per CTA whose candidates the CTA sets up together.

The tuner renders the workload with every candidate, checks that all candidates produce
the same image within 1e-5, times each with CUDA events (median of `reps`), and caches the
winner in a JSON file keyed by (GPU name, resolution bucket, quad-count bucket, colour
mode). The cache path is $LR_AUTOTUNE_CACHE, else ~/.cache/lucidraster_gb300/autotune.json.
"""
from __future__ import annotations

import json
import math
import os
import statistics

import torch

DEFAULT_KS = (1, 2, 3, 4, 6, 8)


def cache_path() -> str:
    p = os.environ.get("LR_AUTOTUNE_CACHE")
    if p:
        return p
    return os.path.join(os.path.expanduser("~"), ".cache", "lucidraster_gb300", "autotune.json")


def workload_key(width: int, height: int, num_quads: int, color_mode: int, device=None) -> str:
    name = torch.cuda.get_device_name(device)
    px = width * height
    return f"{name}|px2^{int(round(math.log2(max(px, 1))))}|q2^{int(round(math.log2(max(num_quads, 1))))}|c{color_mode}"


def _load_cache():
    try:
        with open(cache_path()) as f:
            return json.load(f)
    except Exception:
        return {}


def _save_cache(c):
    p = cache_path()
    os.makedirs(os.path.dirname(p), exist_ok=True)
    tmp = p + f".{os.getpid()}.tmp"
    with open(tmp, "w") as f:
        json.dump(c, f, indent=1, sort_keys=True)
    os.replace(tmp, p)


def lookup(width, height, num_quads, color_mode, device=None):
    return _load_cache().get(workload_key(width, height, num_quads, color_mode, device))


def tune(scene, width: int, height: int, ks=DEFAULT_KS, ctas_per_sm=(0,), reps: int = 5,
         use_cache: bool = True, device=None, carry=None, bin_sizes=(32,), block_hs=(4,), shared=(False,)):
    """scene: a DeviceScene. Returns {'sorter_k', 'raster_ctas_per_sm', 'carry_colors',
    'bin_size', 'block_h', 'ms', 'table'}. carry: candidates for carrying flat colours in the
    sorter (default: both for flat-colour scenes). bin_sizes: candidate bin sizes (16, 32,
    64). block_hs: values of lr_config.block_h (4 and 8 take the same kernels, so a candidate is
    rendered and timed once for both and the choice is 4 where that is among them; 8 is listed
    for sorter capacities up to 3). shared: whether a CTA sets candidates up once per 32x8
    strip (lr_config.shared_setup; 32-pixel bins, 8x4 half-blocks, capacities up to 3)."""
    from . import Renderer
    key = workload_key(width, height, scene.num_quads, scene.color_mode, device)
    cache = _load_cache() if use_cache else {}
    if use_cache and key in cache:
        return cache[key]
    table = []
    ref_img = None
    if carry is None:
        carry = (False, True) if scene.color_mode == 0 else (False,)
    cands = [(k, c, cc, bs, bh, sh) for sh in shared for bh in block_hs for bs in bin_sizes for k in ks
             for c in ctas_per_sm for cc in carry
             if (bh == 4 or k <= 3) and (not sh or (bs == 32 and bh == 4 and k <= 3))]
    measured = {}
    for k, c, cc, bs, bh, sh in cands:
        if (k, c, cc, bs, sh) not in measured:
            r = Renderer(sorter_k=k, raster_ctas_per_sm=c, device=device, carry_colors=cc, bin_size=bs,
                         block_h=bh, shared_setup=sh)
            out = r.make_outputs(width, height)
            view = r.view_struct(scene, width, height, out)
            st = r.render_views([view])                    # sizes the workspace, checked
            img = out["rgba"].clone()
            if ref_img is None:
                ref_img = img
            elif float((img - ref_img).abs().max()) > 1e-5:
                raise RuntimeError(f"sorter_k={k} changed the image beyond 1e-5: the pipeline must be exact")
            times = []
            for _ in range(reps):
                a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
                a.record()
                r.render_views([view], check=False)
                b.record()
                torch.cuda.synchronize()
                times.append(a.elapsed_time(b))
            measured[k, c, cc, bs, sh] = dict(ms=statistics.median(times), overflow_pixels=B_overflow(r),
                                              fragments=int(st.fragments))
            r.close()
        table.append(dict(sorter_k=k, raster_ctas_per_sm=c, carry_colors=cc, bin_size=bs, block_h=bh,
                          shared_setup=sh, **measured[k, c, cc, bs, sh]))
    best = min(table, key=lambda t: (t["ms"], t["block_h"]))
    result = dict(sorter_k=best["sorter_k"], raster_ctas_per_sm=best["raster_ctas_per_sm"],
                  carry_colors=best["carry_colors"], bin_size=best["bin_size"], block_h=best["block_h"],
                  shared_setup=best["shared_setup"],
                  ms=best["ms"], table=table)
    if use_cache:
        cache[key] = result
        _save_cache(cache)
    return result


def B_overflow(r) -> int:
    from . import _binding as B
    return int(B.lr_get_stats(r.ctx, raise_on_error=False).overflow_pixels)
