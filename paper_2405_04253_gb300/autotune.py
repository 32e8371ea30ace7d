"""Launch-shape autotuner for libfnt's transform kernels.

Times each candidate (CDC warps per CTA; AEQ warps per CTA with a cap on the
AEQ warps resident per SM) on a prepared batch with CUDA events around each
stage on the launching stream, after warm-up, and keeps the fastest per stage.
Only stages whose kernel has these settings are tuned: the direct forms, which a
plan runs unless it picks a transform kernel, have shapes of their own, and so have
the kernels that a plan picks with set_cdc_kernel(2) and set_aeq_kernel(2).  Results
are cached in a JSON file keyed by the workload's shape and the tuned stages, so a
later run with the same shape reuses them.  Only launch shapes change: results are
bit-identical for every candidate.
"""
from __future__ import annotations

import json
import os

from . import OP_AEQ, OP_CDC, OP_CHAIN, Batch, Plan

CANDIDATES = (1, 2, 3, 4)
_SRC_TAG = None


def _src_tag() -> str:
    """Short hash of the library's sources: a cache entry written by another
    build of the kernels is not reused."""
    global _SRC_TAG
    if _SRC_TAG is None:
        import hashlib
        csrc = os.path.join(os.path.dirname(os.path.abspath(__file__)), "csrc")
        h = hashlib.sha256()
        for name in sorted(os.listdir(csrc)):
            with open(os.path.join(csrc, name), "rb") as fh:
                h.update(name.encode() + fh.read())
        _SRC_TAG = h.hexdigest()[:12]
    return _SRC_TAG
OCCUPANCY = (0, 12, 16, 20)          # AEQ warps per SM cap (0: none)


def tunable(plan: Plan, op: int) -> tuple:
    """The stages of `op` ("cdc", "aeq") whose kernels have launch settings."""
    stages = []
    # asked for work that fills the GPU: smaller work may take another transform kernel
    # (also on a plan that picks none: aeq_freq_sum = 1)
    if op != OP_AEQ and plan.cdc_route(1 << 20) == "cdc_kernel":
        stages.append("cdc")
    if op != OP_CDC and plan.aeq_route(1 << 20, 1 << 20, 1) == "aeq_kernel":
        stages.append("aeq")
    return tuple(stages)


def _key(plan: Plan, frames, op: int, stages=("cdc", "aeq")) -> str:
    d = plan.desc
    lens = sorted(int(f.n) for f in frames)
    total = sum(lens)
    return (f"op{op}_n{len(frames)}_tot{total}_max{lens[-1] if lens else 0}_aeq{d.n_aeq}"
            f"_seg{d.aeq_segment}_{d.aeq_warmup}_p{d.aeq_update_period}_{'_'.join(stages)}_src{_src_tag()}")


def _time_stage(batch: Batch, stage: int, reps: int, stream) -> float:
    import torch
    evs = [torch.cuda.Event(enable_timing=True) for _ in range(2)]
    for _ in range(2):
        batch.launch_stage(stage, stream)
    evs[0].record(stream)
    for _ in range(reps):
        batch.launch_stage(stage, stream)
    evs[1].record(stream)
    torch.cuda.synchronize()
    return evs[0].elapsed_time(evs[1]) / reps


def _apply(plan: Plan, best: dict):
    if "cdc" in best["tuned"]:
        plan.set_launch(cdc_warps=best["cdc_warps"])
    if "aeq" in best["tuned"]:
        plan.set_launch(aeq_warps=best["aeq_warps"])
        plan.set_aeq_occupancy(best["aeq_occupancy"])


def tune(plan: Plan, frames, op: int = OP_CHAIN, reps: int = 20, cache: str | None = None) -> dict:
    """Picks and applies the fastest launch shape for each stage of `op` on
    these frames that can be tuned; returns {"tuned": those stages, "cdc_warps",
    "aeq_warps", "aeq_occupancy", "cdc_ms", "aeq_ms"}.  A stage that cannot be tuned
    is timed once, as it runs, and the plan's settings for it are left alone."""
    import torch
    stages = tunable(plan, op)
    key = _key(plan, frames, op, stages)
    if cache and stages and os.path.exists(cache):
        try:
            with open(cache) as fh:
                hit = json.load(fh).get(key)
        except (OSError, ValueError):
            hit = None
        if hit:
            _apply(plan, hit)
            return hit
    stream = torch.cuda.current_stream()
    batch = Batch(plan, frames, op, use_graph=False)
    best = {"tuned": list(stages), "cdc_warps": 4, "aeq_warps": 2, "aeq_occupancy": 0}
    for stage, name in ((0, "cdc"), (1, "aeq")):
        if op == (OP_AEQ, OP_CDC)[stage]:
            continue
        if name not in stages:
            best[name + "_ms"] = _time_stage(batch, stage, reps, stream)
            continue
        for w in CANDIDATES:
            for occ in (OCCUPANCY if stage == 1 else (0,)):
                if stage == 0:
                    plan.set_launch(cdc_warps=w)
                else:
                    if occ and occ < w:
                        continue
                    plan.set_launch(aeq_warps=w)
                    plan.set_aeq_occupancy(occ)
                ms = _time_stage(batch, stage, reps, stream)
                if name + "_ms" not in best or ms < best[name + "_ms"]:
                    best[name + "_ms"] = ms
                    best[name + "_warps"] = w
                    if stage == 1:
                        best["aeq_occupancy"] = occ
    _apply(plan, best)
    batch.close()
    if cache and stages:
        data = {}
        if os.path.exists(cache):
            try:
                with open(cache) as fh:
                    data = json.load(fh)
            except (OSError, ValueError):
                data = {}
        data[key] = best
        tmp = cache + f".tmp{os.getpid()}"
        with open(tmp, "w") as fh:
            json.dump(data, fh, indent=1)
        os.replace(tmp, cache)
    return best
