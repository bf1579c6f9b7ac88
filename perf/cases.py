"""The work that users of this library have it do, as cases that can be timed and compared.

Every case goes through the public Python entry points (paper_1705_01813_gb300.gkm) with data shaped like the
repository's workloads: Gaussian mixtures (the plain method and the serving jobs), SIFT-shaped integers, GIST-shaped
values in [0, 1] and deep-feature-shaped unit vectors in bfloat16.  Whole graph constructions and fits stand beside
the single steps a custom loop calls (assignment, update), the quality estimate, the paper's initial partition, the
boost form and a batch of serving jobs.

listed() names the cases, draw(rng) gives another case of the same ranges, prepare(case, seed) makes what a program
holds before the call, run(state) is one pass, work(case) is the traffic and arithmetic no implementation avoids, and
exact(case, seed) gives the computed numbers in 64 bits where plain torch can.
"""
from __future__ import annotations

import math
import random

import torch

from paper_1705_01813_gb300 import datagen, gkm

SCREEN4 = 4 | (4 << 8)  # int8 screening of the candidates, four per group: the tuner's choice for wide rows


def listed():
    return [
        # the smallest fit: the plain method's Gaussian workload, where launches and latency count
        dict(name="fit_gauss_20k", op="fit", data="gauss", n=20_000, d=32, k=200, kappa=20, iters=10, bf16=False,
             precision=1),
        # the graph for it
        dict(name="build_gauss_20k", op="build", data="gauss", n=20_000, d=32, k=200, kappa=20, tau=10, bf16=False,
             precision=1),
        # the graph of a SIFT-sized descriptor set (FP32 integers), the paper's best-known workload
        dict(name="build_sift_1m", op="build", data="sift", n=1_000_000, d=128, k=10_000, kappa=50, tau=10, bf16=False,
             precision=1),
        # the graph of wide FP32 descriptors (GIST-shaped)
        dict(name="build_gist_200k", op="build", data="gist", n=200_000, d=960, k=2_000, kappa=50, tau=10, bf16=False,
             precision=SCREEN4),
        # the graph and the fit of deep features stored in bfloat16, with very many small clusters
        dict(name="build_deep_2m", op="build", data="deep", n=2_000_000, d=512, k=200_000, kappa=40, tau=10, bf16=True,
             precision=SCREEN4),
        dict(name="fit_deep_2m", op="fit", data="deep", n=2_000_000, d=512, k=200_000, kappa=40, iters=10, bf16=True,
             precision=SCREEN4),
        # single steps of a custom loop: the SIFT-shaped assignment, and an update at ragged sizes
        dict(name="assign_sift_1m", op="assign", data="sift", n=1_000_000, d=128, k=10_000, kappa=50, bf16=False,
             precision=1),
        dict(name="update_ragged_300k", op="update", data="gauss", n=300_007, d=100, k=3_001, kappa=20, bf16=False,
             precision=1),
        # serving: jobs of one width that wait together run as one batch
        dict(name="batch_16_jobs_d64", op="batch", data="gauss", jobs=16, n_lo=10_000, n_hi=200_000, job_seed=3, d=64,
             kappa=20, tau=10, iters=10, bf16=False, precision=1),
        # graph quality on sampled queries (top-1 recall), the paper's initial partition, the boost form's moves
        dict(name="recall_sift_1m", op="recall", data="sift", n=1_000_000, d=128, k=10_000, kappa=50, queries=1_000,
             bf16=False, precision=1),
        dict(name="tree_sift_1m", op="tree", data="sift", n=1_000_000, d=128, k=10_000, kappa=50, iters=2, bf16=False,
             precision=1),
        dict(name="boost_sift_1m", op="boost", data="sift", n=1_000_000, d=128, k=10_000, kappa=50, visits=20_000,
             bf16=False, precision=1),
    ]


def _log_uniform(rng: random.Random, lo: int, hi: int) -> int:
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng: random.Random):
    """A case of the listed kinds at other sizes: n over the range of each kind, narrow and wide rows (some of odd
    width), few large and many small clusters, both sample types and the precision levels users choose."""
    op = rng.choice(["fit", "build", "fit", "build", "assign", "assign", "update", "update", "batch", "recall",
                     "tree", "boost"])
    bf16 = rng.random() < 0.4
    d = rng.choice([24, 32, 33, 48, 64, 72, 96, 100, 128, 128, 160, 200, 256, 300, 384, 512, 768, 960])
    top = {"fit": 1_500_000, "build": 1_200_000, "assign": 2_000_000, "update": 2_000_000, "recall": 1_000_000,
           "tree": 1_000_000, "boost": 1_000_000, "batch": 200_000}[op]
    n = _log_uniform(rng, 5_000, max(6_000, min(top, int(2.0e8 / d))))
    per = _log_uniform(rng, 10, 200)  # samples per cluster
    kappa = rng.choice([10, 20, 20, 32, 40, 50])
    if bf16:
        data = "deep" if d >= 256 else rng.choice(["gauss", "sift"])
    else:
        data = "gist" if d >= 768 else rng.choice(["gauss", "sift"])
    precision = rng.choice([0, 1, 1, 1, 4, SCREEN4]) if d <= 256 else rng.choice([1, 4, SCREEN4, SCREEN4])
    c = dict(op=op, data=data, n=n, d=d, k=max(2, n // per), kappa=kappa, bf16=bf16, precision=precision)
    if op == "fit":
        c.update(iters=10)
    elif op == "build":
        c.update(tau=10)
    elif op == "batch":
        c = dict(op=op, data="gauss", jobs=rng.randint(2, 24), n_lo=10_000, n_hi=max(12_000, min(200_000, n)),
                 job_seed=rng.randint(0, 1 << 20), d=rng.choice([64, 128, 256]), kappa=20, tau=10, iters=10,
                 bf16=False, precision=rng.choice([0, 1, 1, 2]))
        c["jobs"] = min(c["jobs"], max(2, int(9.0e7 / (c["d"] * c["n_hi"]))))
    elif op == "recall":
        c.update(queries=rng.choice([100, 500, 1_000]))
    elif op == "tree":
        c.update(iters=rng.choice([1, 2, 2]))
        if d > 512:
            c.update(d=128, data="sift")
    elif op == "boost":
        c.update(visits=min(n, rng.choice([2_000, 5_000, 10_000])))
        if d > 512:
            c.update(d=100, data="sift")
    return c


# --------------------------------------------------------------------------------------------------------------
# Inputs
# --------------------------------------------------------------------------------------------------------------
def _gen(seed: int) -> torch.Generator:
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed))
    return g


def _samples(data: str, n: int, d: int, bf16: bool, seed: int) -> torch.Tensor:
    """n x d samples of one of the workload shapes, drawn on the device."""
    latent = max(8, n // 100)
    if data == "deep":  # unit vectors around weakly concentrated directions
        X = datagen.deep_like_device(n, d, n_dirs=max(16, n // 5), kappa_vmf=50.0, seed=seed)
        return X if bf16 else X.float()
    if data == "gauss":  # isotropic mixture, centres in [-10, 10]^d
        X = datagen.gauss_mixture_device(n, d, latent, seed, "cuda")
        return X.to(torch.bfloat16) if bf16 else X
    g = _gen(seed)
    X = torch.empty((n, d), dtype=torch.bfloat16 if bf16 else torch.float32, device="cuda")
    if data == "sift":  # integers 0..255, log-normal around latent centres, mean about 20
        mu = torch.randn((latent, d), generator=g, device="cuda") * 0.5 + (math.log(20.0) - 0.37)
    else:  # gist: values in [0, 1] around latent centres of mean 0.2
        mu = (torch.rand((latent, d), generator=g, device="cuda") ** 2 * 0.6).clamp(1e-3, 1 - 1e-3)
    step = 1 << 17
    for s in range(0, n, step):
        m = min(n, s + step) - s
        c = mu[torch.randint(0, mu.shape[0], (m,), generator=g, device="cuda")]
        e = torch.randn((m, d), generator=g, device="cuda")
        if data == "sift":
            X[s:s + m] = torch.exp(c + 0.7 * e).round().clamp(0, 255)
        else:
            X[s:s + m] = (c + torch.sqrt(c * (1 - c) / 51.0) * e).clamp(0, 1)
    return X


def _batch_jobs(case, seed: int):
    """(n, k, graph seed, fit seed) of each job: n log-uniform, k = n / 100."""
    r = random.Random(case["job_seed"])
    ns = [_log_uniform(r, case["n_lo"], case["n_hi"]) for _ in range(case["jobs"])]
    return [(n, max(1, n // 100), seed * 64 + j, seed * 64 + j + 7) for j, n in enumerate(ns)]


def prepare(case, seed):
    """What a program holds before the call: samples, and for the later steps the graph and the partition that the
    earlier ones gave it."""
    op, kappa = case["op"], case["kappa"]
    s = dict(case=case, seed=int(seed))
    if op == "batch":
        jobs = _batch_jobs(case, int(seed))
        s["jobs"] = jobs
        s["X"] = torch.cat([_samples("gauss", n, case["d"], case["bf16"], int(seed) * 64 + j)
                            for j, (n, _, _, _) in enumerate(jobs)])
        return s
    n, d, k = case["n"], case["d"], case["k"]
    X = _samples(case["data"], n, d, case["bf16"], int(seed))
    s["X"] = X
    g = _gen(int(seed) + 1)
    if op in ("fit", "assign", "recall", "boost"):
        s["gi"], _, _, _ = gkm.build_knn_graph(X, kappa, tau=4, seed=int(seed), want_log=False, precision=1)
    if op == "fit":
        s["labels"] = torch.randint(0, k, (n,), generator=g, device="cuda", dtype=torch.int32)
    elif op == "assign":  # the state in the middle of a fit
        L0 = torch.randint(0, k, (n,), generator=g, device="cuda", dtype=torch.int32)
        s["labels"], s["C"], _, _ = gkm.kmeans_fit(X, k, s["gi"], 3, init_labels=L0, want_log=False, precision=1)
    elif op == "update":  # clusters of uneven size, a few of them empty
        z = torch.rand(n, generator=g, device="cuda") ** 1.5
        s["labels"] = (z * k).to(torch.int32).clamp(0, k - 1)
        s["C"] = torch.zeros((k, d), dtype=torch.float32, device="cuda")
    elif op == "recall":
        s["queries"] = torch.randint(0, n, (case["queries"],), generator=g, device="cuda", dtype=torch.int32)
    elif op == "boost":
        L0 = torch.randint(0, k, (n,), generator=g, device="cuda", dtype=torch.int32)
        s["labels"], _, _, _ = gkm.kmeans_fit(X, k, s["gi"], 5, init_labels=L0, want_log=False, precision=1)
        s["D"], s["counts"], s["S"] = gkm.boost_init(X, s["labels"], k)
        s["order"] = torch.randperm(n, generator=g, device="cuda")[:case["visits"]].to(torch.int32)
    return s


# --------------------------------------------------------------------------------------------------------------
# One pass
# --------------------------------------------------------------------------------------------------------------
def run(state):
    case, X = state["case"], state["X"]
    op = case["op"]
    if op == "build":
        return gkm.build_knn_graph(X, case["kappa"], tau=case["tau"], seed=state["seed"],
                                   precision=case["precision"])
    if op == "fit":
        return gkm.kmeans_fit(X, case["k"], state["gi"], case["iters"], init_labels=state["labels"],
                              precision=case["precision"])
    if op == "assign":
        return gkm.assign_step(X, state["gi"], state["C"], state["labels"], precision=case["precision"])
    if op == "update":
        return gkm.update_step(X, state["labels"], case["k"], state["C"])
    if op == "batch":
        return gkm.batch_fit(X, state["jobs"], case["kappa"], tau=case["tau"], iters=case["iters"],
                             precision=case["precision"])
    if op == "recall":
        return gkm.graph_recall(X, state["gi"], state["queries"])
    if op == "tree":
        return gkm.two_means_tree(X, case["k"], iters=case["iters"], seed=state["seed"])
    # boost: the epoch moves samples in place, from the partition the program keeps
    L, D = state["labels"].clone(), state["D"].clone()
    counts, S = state["counts"].clone(), state["S"].clone()
    moved = gkm.boost_epoch(X, state["gi"], state["order"], L, case["k"], D, counts, S)
    return L, D, counts, S, moved


# --------------------------------------------------------------------------------------------------------------
# What a pass cannot do without
# --------------------------------------------------------------------------------------------------------------
def work(case):
    """Inputs read once per pass over the samples, outputs written once; distances of d terms count 3 d operations.
    A graph round or fit iteration needs the samples once.  About half of the kappa + 1 candidate clusters of a
    sample are distinct; a graph round compares the pairs inside clusters of 50."""
    op, d, es, kappa = case["op"], case["d"], 2 if case["bf16"] else 4, case["kappa"]
    u = (kappa + 1) / 2
    if op == "batch":
        jobs = _batch_jobs(case, 0)
        n, k = sum(j[0] for j in jobs), sum(j[1] for j in jobs)
        rounds = case["tau"] + case["iters"]
        return {"bytes": float((rounds + 1) * n * d * es + n * (8 * kappa + 4) + 4 * k * d),
                "flops": float(3 * d * n * (kappa + rounds * u + case["tau"] * 24.5))}
    n, k = case["n"], case["k"]
    x, graph = n * d * es, 4 * n * kappa
    if op == "build":
        return {"bytes": float((case["tau"] + 1) * x + 2 * graph + 4 * n),
                "flops": float(3 * d * n * (kappa + case["tau"] * (u + 24.5)))}
    if op == "fit":
        return {"bytes": float((case["iters"] + 1) * x + case["iters"] * graph + 8 * n + 4 * k * d),
                "flops": float(case["iters"] * 3 * d * n * u)}
    if op == "assign":
        return {"bytes": float(x + graph + 12 * n + 4 * k * d), "flops": float(3 * d * n * u)}
    if op == "update":
        return {"bytes": float(x + 8 * n + 4 * k * d + 8 * k), "flops": float(2 * d * n)}
    if op == "recall":
        return {"bytes": float(x + 12 * case["queries"]), "flops": float(3 * d * n * case["queries"])}
    if op == "tree":  # every depth of the tree reads the samples for each 2-means pass and for the split
        depth = max(1, math.ceil(math.log2(max(2, k))))
        return {"bytes": float(depth * (case["iters"] + 1) * x + 4 * n),
                "flops": float(depth * (case["iters"] + 1) * 6 * d * n)}
    m = case["visits"]
    return {"bytes": float(m * (d * es + 8 * kappa + u * 8 * d) + 24 * k * d),
            "flops": float(m * (u + 1) * 3 * d)}


# --------------------------------------------------------------------------------------------------------------
# The computed numbers in 64 bits, by plain torch
# --------------------------------------------------------------------------------------------------------------
def _assign64(X, gi, C, L):
    """Labels and squared distances of the nearest candidate centroid (ties to the smaller label)."""
    n, d = X.shape
    out, best = torch.empty_like(L), torch.empty(n, dtype=torch.float64, device=X.device)
    step = max(256, int(6e8 / (8 * d * (gi.shape[1] + 1))))
    for s in range(0, n, step):
        e = min(n, s + step)
        lab = torch.cat([L[s:e, None], L[gi[s:e].long()]], 1).long()
        lab, _ = lab.sort(1)  # ascending labels: the first minimum is the smaller label
        diff = X[s:e, None, :].double() - C[lab]
        d2 = (diff * diff).sum(2)
        best[s:e], j = d2.min(1)
        out[s:e] = lab.gather(1, j[:, None])[:, 0].to(torch.int32)
    return out, best


def _means64(X, L, k, C):
    """Centroids (an empty cluster keeps its row of C), sizes and the summed squared distance to them."""
    n, d = X.shape
    cnt = torch.bincount(L.long(), minlength=k)
    S = torch.zeros((k, d), dtype=torch.float64, device=X.device)
    step = 1 << 18
    for s in range(0, n, step):
        S.index_add_(0, L[s:s + step].long(), X[s:s + step].double())
    C = torch.where(cnt[:, None] > 0, S / cnt.clamp(min=1)[:, None], C)
    tot = torch.zeros((), dtype=torch.float64, device=X.device)
    for s in range(0, n, step):
        diff = X[s:s + step].double() - C[L[s:s + step].long()]
        tot += (diff * diff).sum()
    return C, cnt, tot


def exact(case, seed):
    op = case["op"]
    if op in ("build", "batch", "tree", "boost"):  # whole numbers, or results that follow from many decisions
        return None
    s = prepare(case, seed)
    X, n = s["X"], case["n"]
    if op == "fit":
        if n * case["d"] * case["kappa"] * case["iters"] > 2.5e10:
            return None
        L = s["labels"]
        C, cnt, tot = _means64(X, L, case["k"], torch.zeros((case["k"], case["d"]), dtype=torch.float64,
                                                            device=X.device))
        log = [float(tot) / n]
        for _ in range(case["iters"]):
            L, best = _assign64(X, s["gi"], C, L)
            log.append(float(best.sum()) / n)
            C, cnt, tot = _means64(X, L, case["k"], C)
            log.append(float(tot) / n)
        return None, C, None, log
    if op == "assign":
        _, best = _assign64(X, s["gi"], s["C"].double(), s["labels"])
        return None, best, best.sum()[None], None
    if op == "update":
        C, _, tot = _means64(X, s["labels"], case["k"], s["C"].double())
        return C, None, tot[None], None, None
    # recall: the nearest other sample of every query
    q = s["queries"].long()
    best = torch.full((q.numel(),), math.inf, dtype=torch.float64, device=X.device)
    Q = X[q].double()
    step = max(1024, int(1e9 / (8 * q.numel())))
    for a in range(0, n, step):
        b = min(n, a + step)
        d2 = torch.cdist(Q, X[a:b].double(), compute_mode="donot_use_mm_for_euclid_dist") ** 2
        own = (q >= a) & (q < b)
        d2[own.nonzero()[:, 0], q[own] - a] = math.inf
        best = torch.minimum(best, d2.min(1).values)
    return None, None, best
