"""Autotuner over the library's precision levels and the assignment's tile shape.

Every level gives the same labels, centroids, distortions and graph bit for bit (the GPU tests assert it), so
the fastest one for a workload can be chosen by measurement alone.  Timed with CUDA events on the caller's samples and
graph, per level (0 to 4; 3 only for FP32 samples): a whole fit of `iters` iterations from seeded labels, as an
iteration inside a fit costs less than an assignment by itself at all levels but 3 (they evaluate only what the
previous iteration can have changed); one assignment; and one refinement per refinement path (level 0: the FP32 tiles;
levels 1 to 4: the tensor-core Gram where d allows it).  A level's score is the time of its fit's iterations, tau +
iters of them (a graph construction runs one per round), and of tau refinements.  Where the assignment's kernel reads
its candidates in groups of 4 or of 8 (bits 8-15 of the precision argument: FP32 and BF16 rows of more than 64 and at
most 512 values; the kernels' summation tree is the same for both, so the results are too) the assignment is timed
with both, and the faster width goes with the level.  Choices are cached per shape key.
"""
from __future__ import annotations

import torch

from . import gkm

_CACHE: dict = {}


def _bucket(v: int) -> int:
    """Powers of two: shapes within a factor of two share a tuning."""
    return max(1, int(v)).bit_length()


def shape_key(X: torch.Tensor, k: int, kappa: int) -> tuple:
    props = torch.cuda.get_device_properties(X.device)
    return (props.name, str(X.dtype), int(X.shape[1]), int(kappa), _bucket(X.shape[0]), _bucket(k))


def _time(fn, reps: int) -> float:
    fn()
    best = float("inf")
    for _ in range(reps):
        a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        a.record()
        fn()
        b.record()
        b.synchronize()
        best = min(best, a.elapsed_time(b))
    return best


def _widths(p: int, d: int) -> list:
    """Candidates per group worth timing at level p: [0], the default, where the kernel does not read them (level 3, the
    int8 screening, FP32 rows of at most 64 values) or has one form (rows of more than 512 values)."""
    if p in (3, 4) or d > 512 or (p <= 1 and d <= 64) or (p == 1 and d > 288):
        return [0]
    return [8, 4]


def tune_precision(X: torch.Tensor, g_idx: torch.Tensor, g_dist: torch.Tensor, labels: torch.Tensor, k: int,
                   tau: int = 10, iters: int = 10, max_cluster: int = 128, reps: int = 3,
                   use_cache: bool = True) -> dict:
    """Fastest precision level for the samples X with graph (g_idx, g_dist) and labels at k clusters.

    The graph and labels are read, never changed (the refinement is timed on copies).  Returns
    {"precision": p, "assign_ms": {p: ms}, "fit_ms": {p: ms}, "refine_ms": {path: ms}, "score_ms": {p: ms}, "key": key}.
    """
    kappa = g_idx.shape[1]
    key = shape_key(X, k, kappa)
    if use_cache and key in _CACHE:
        return _CACHE[key]
    n, d = X.shape
    dev = X.device
    levels = [0, 1, 2, 4] if X.dtype == torch.bfloat16 else [0, 1, 2, 3, 4]
    off, mem, cnt = gkm.group_by_label(labels, k)
    C = torch.zeros((k, d), dtype=torch.float32, device=dev)
    gkm.update_from_groups(X, off, mem, k, C, cnt)
    ws = gkm.workspace(max(gkm.workspace_size(op, n, d, k, kappa)
                           for op in (gkm.GK_OP_ASSIGN, gkm.GK_OP_REFINE, gkm.GK_OP_FIT)), dev)
    out = torch.empty_like(labels)
    assign_ms, fit_ms, group_width = {}, {}, {}
    fit_iters = max(1, iters)
    for p in levels:
        best_w, best_t = 0, float("inf")
        for gw in _widths(p, d):
            code = p | (gw << 8)
            t = _time(lambda: gkm.assign_step(X, g_idx, C, labels, out, None, None, None, code, mem, ws=ws), reps)
            if t < best_t:
                best_w, best_t = gw, t
        assign_ms[p], group_width[p] = best_t, best_w
    for p in levels:
        code = p | (group_width[p] << 8)
        fit_ms[p] = _time(lambda: gkm.kmeans_fit(X, k, g_idx, fit_iters, seed=1, labels_out=out, C_out=C, counts_out=cnt,
                                                 want_log=False, precision=code, ws=ws), 1)
    gi, gd = g_idx.clone(), g_dist.clone()

    def refine(p):
        gi.copy_(g_idx)
        gd.copy_(g_dist)
        gkm.graph_refine_groups(X, off, mem, k, gi, gd, max_cluster, p, ws=ws)

    refine_ms = {"fp32_tiles": _time(lambda: refine(0), reps), "precision_ge_1": _time(lambda: refine(1), reps)}
    copy_ms = _time(lambda: (gi.copy_(g_idx), gd.copy_(g_dist)), reps)
    score = {p: fit_ms[p] / fit_iters * (tau + iters) +
             (refine_ms["fp32_tiles"] if p == 0 else refine_ms["precision_ge_1"]) * tau - copy_ms * tau
             for p in levels}
    best = min(levels, key=lambda p: (score[p], p))
    res = {"precision": best | (group_width[best] << 8), "level": best, "group_width": group_width[best],
           "assign_ms": assign_ms, "fit_ms": fit_ms, "group_width_by_level": group_width, "refine_ms": refine_ms,
           "score_ms": score, "key": list(key)}
    _CACHE[key] = res
    return res
