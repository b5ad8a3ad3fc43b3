"""Autotuner for the batched (graph-captured) launch.

A launch's schedule has two kinds of free parameters:
  * the plan: how many events the UNet processes per pass (chunk_events). Small chunks
    keep a pass's activations resident in the 129 MB L2 and shrink the pool; large chunks
    give each layer kernel more tiles per SM and fewer launches;
  * the grids: how many CTAs per SM each persistent kernel family launches (pvf_schedule:
    the front, whose grid sets the events each CTA walks and, in the tensor-core forms,
    the FC tile (passes of 256 tracks at 1-2 CTAs per SM, 128 at 3-4), the tensor-core conv
    kernels, whose grids set the tiles per CTA, and the peak finder). More resident CTAs
    hide latency; fewer leave each CTA more shared-memory and register headroom and
    shorten the tail of the last wave. Only values that change a launch are tried
    (grid_candidates): a measured difference between two equal launches is noise.
For a workload the tuner captures the whole batch as one CUDA graph per candidate, times
graph launches with CUDA events (L2 flushed between launches), and walks the parameters
one at a time (coordinate descent), keeping each parameter at its fastest value before
moving to the next. The result is a table of the schedule plus every trial, which
PVFinder(schedule=...) and pvf_create read; results never depend on the schedule.
"""

from __future__ import annotations

import json
import os

FAMILIES = ("front", "enc2", "enc3", "enc4_up3", "dec3_up2", "dec2_up1", "dec1_final", "tail")
# CTAs per SM tried for each family, by form and UNet base width, beside 0 (as many as fit): those
# values that are below what fits an SM. Families left out have no kernel of their own (the encoder
# of whole events at width 16 is one kernel of one CTA per SM; the float32 form has no conv entries)
# or only one CTA that fits.
_FRONT = (1, 2, 3, 4)           # 1-2 and 3-4 are two shapes of the kernel
GRID_CANDIDATES = {
    ("fp32", 16): {"front": (1,), "tail": (1,)},
    ("fp32", 32): {"front": (1,), "tail": (1,)},
    ("16-bit", 16): {"front": _FRONT, "dec2_up1": (1,), "dec1_final": (1,), "tail": (1, 2)},
    ("16-bit", 32): {"front": _FRONT, "enc2": (2, 3), "tail": (1, 2)},
    ("fp8", 16): {"front": _FRONT, "dec3_up2": (1,), "dec2_up1": (1, 2), "dec1_final": (1,), "tail": (1, 2)},
    ("fp8", 32): {"front": _FRONT, "enc2": (2, 3), "enc3": (1,), "enc4_up3": (1,), "dec3_up2": (1,), "dec2_up1": (1,),
                  "tail": (1, 2)},
}
TUNED_DIR = os.path.join(os.path.dirname(os.path.abspath(__file__)), "tuned")


def grid_candidates(precision, width):
    """{family: CTAs per SM to try} for whole events of this form and UNet base width."""
    return GRID_CANDIDATES["16-bit" if precision in ("bf16", "fp16") else precision, width]


def _time_graph(pv, feats, offs, repeats, warmup, flush):
    import torch
    out = pv.alloc_outputs(int(offs.numel() - 1))
    g = pv.capture_graph(feats, offs, out)
    for _ in range(warmup):
        g.launch()
    times = []
    for _ in range(repeats):
        flush.fill_(1)
        a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        a.record()
        g.launch()
        b.record()
        torch.cuda.synchronize()
        times.append(a.elapsed_time(b))
    g.close()
    return min(times)


def tune(weights, batch, precision="bf16", chunk_candidates=(0,), repeats=3, warmup=1, max_pv=64,
         fp8_act_scales=None, flush_mb=512, passes=1, log=None):
    """Coordinate descent over chunk_events and the CTAs per SM of each kernel family.
    Returns (best: dict with "chunk_events" and the schedule, trials: list of dicts)."""
    import torch
    from .pvf import PVFinder
    from .weights import unet_width

    n = batch.n_events
    feats = torch.from_numpy(batch.features).cuda()
    offs = torch.from_numpy(batch.offsets).cuda()
    flush = torch.empty(flush_mb * 1024 * 1024, dtype=torch.uint8, device="cuda")
    trials = []
    cache = {}

    def measure(chunk, sched):
        key = (chunk, tuple(sorted(sched.items())))
        if key in cache:
            return cache[key]
        pv = PVFinder(weights, precision=precision, max_events=n, chunk_events=min(chunk, n) if chunk else 0,
                      max_pv_per_event=max_pv, fp8_act_scales=fp8_act_scales, schedule=sched)
        ms = _time_graph(pv, feats, offs, repeats, warmup, flush)
        pv.close()
        del pv
        torch.cuda.empty_cache()
        trials.append({"chunk_events": chunk, **sched, "ms": ms})
        if log:
            log(f"chunk {chunk or n} {sched}: {ms:.3f} ms")
        cache[key] = ms
        return ms

    chunk, sched = 0, {f: 0 for f in FAMILIES}
    best_ms = measure(chunk, sched)
    for _ in range(passes):
        for c in chunk_candidates:
            ms = measure(c, sched)
            if ms < best_ms:
                best_ms, chunk = ms, c
        for fam, values in grid_candidates(precision, unet_width(weights)).items():
            for v in values:
                cand = dict(sched, **{fam: v})
                ms = measure(chunk, cand)
                if ms < best_ms:
                    best_ms, sched = ms, cand
    best = {"chunk_events": chunk, **sched, "ms": best_ms}
    return best, trials


def table_path(precision: str, workload: str) -> str:
    return os.path.join(TUNED_DIR, f"{precision}_{workload}.json")


def save_table(path, workload: str, precision: str, best: dict, trials: list, default_ms: float):
    os.makedirs(os.path.dirname(path), exist_ok=True)
    with open(path, "w") as fh:
        json.dump({"workload": workload, "precision": precision, "default_ms": default_ms,
                   "best": best, "trials": trials}, fh, indent=1)


def load_schedule(path):
    """(chunk_events, schedule dict) of a saved table."""
    with open(path) as fh:
        best = json.load(fh)["best"]
    return int(best.get("chunk_events", 0)), {f: int(best.get(f, 0)) for f in FAMILIES}
