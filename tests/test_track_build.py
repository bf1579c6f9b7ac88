"""Graph constructions and batches large enough to evaluate only what the previous round's moves can have changed (2^22
sample values and more): a construction must equal the same rounds driven step by step, where every assignment
evaluates all candidates, and a batch its jobs alone, which are below that size; bit for bit."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu

LARGE = 1 << 22


def _samples(n, d, kind, seed):
    g = np.random.default_rng(seed)
    c = max(4, n // 60)
    X = g.uniform(-10, 10, (c, d))[g.integers(0, c, n)] + g.standard_normal((n, d))
    X = torch.from_numpy(X.astype(np.float32)).cuda()
    if kind == "int":
        X = (X * 6 + 64).round().clamp(0, 255)
    if kind == "nan":
        X[17, 3] = float("nan")
    return X.to(torch.bfloat16) if kind == "bf16" else X


@pytest.mark.parametrize("n, d, kind, kappa, max_cluster, precision", [
    (131_072, 32, "f32", 20, 128, 0),        # the smallest size that is tracked
    (127_101, 33, "f32", 16, 64, 0),         # rows that are not 16-byte vectors
    (32_801, 128, "int", 50, 128, 1),        # tensor cores, equal distances
    (66_001, 64, "f32", 20, 128, 1),         # tensor cores, recomputed pairs
    (8_300, 512, "bf16", 40, 128, 4),        # warp-specialised tiles, int8 candidates
    (14_101, 300, "f32", 65, 128, 1),        # int8 candidates at level 1, three row slots
    (4_500, 960, "f32", 50, 128, 0),
    (17_000, 256, "f32", 20, 300, 2),        # runs longer than a tile, BF16 candidates
    (45_001, 96, "nan", 10, 128, 1),         # a non-finite sample
])
def test_construction_equals_rounds(n, d, kind, kappa, max_cluster, precision):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1705_01813_gb300 import gkm
    assert n * d >= LARGE
    X = _samples(n, d, kind, n + d)
    xi, tau = 50, 7
    k0 = max(1, n // xi)
    gi, gd, lab, log = gkm.build_knn_graph(X, kappa, xi=xi, tau=tau, max_cluster=max_cluster, seed=5, precision=precision)
    gi2, gd2 = gkm.init_graph(X, kappa, 5)
    L = gkm.init_labels(n, k0, 5)
    C = torch.zeros((k0, d), device="cuda")
    _, _, e, _, _ = gkm.update_step(X, L, k0, C)
    want = [float(e) / n]
    for _ in range(tau):
        L, _, s, _ = gkm.assign_step(X, gi2, C, L, precision=precision)
        want.append(float(s) / n)
        _, _, e, _, _ = gkm.update_step(X, L, k0, C)
        want.append(float(e) / n)
        gkm.graph_refine(X, L, k0, gi2, gd2, max_cluster=max_cluster, precision=precision)
    gkm.read_status(gkm.workspace(1))  # the calls share this thread's workspace
    assert torch.equal(lab, L)
    assert torch.equal(gi, gi2)
    assert torch.equal(gd.view(torch.int32), gd2.view(torch.int32))
    assert np.array_equal(np.array(log), np.array(want), equal_nan=True)


@pytest.mark.parametrize("d, precision, sizes", [
    (64, 1, [30_000, 20_001, 517, 40_000]),
    (128, 2, [12_000, 64, 30_001]),
    (300, 4, [9_000, 3_000, 5_001]),
])
def test_batch_equals_jobs_alone(d, precision, sizes):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1705_01813_gb300 import gkm
    assert sum(sizes) * d >= LARGE > max(sizes) * d
    kappa, xi, tau, iters = 12, 50, 5, 7
    jobs = [(n, max(1, n // 40), 100 + 3 * j, 101 + 3 * j) for j, n in enumerate(sizes)]
    Xs = [_samples(n, d, "f32", 7 + j) for j, n in enumerate(sizes)]
    gi, gd, lab, C, dist = gkm.batch_fit(torch.cat(Xs), jobs, kappa, xi=xi, tau=tau, iters=iters, precision=precision)
    first = kfirst = 0
    for j, ((n, k, gs, fs), x) in enumerate(zip(jobs, Xs)):
        gi1, gd1, _, _ = gkm.build_knn_graph(x, kappa, xi=xi, tau=tau, seed=gs, want_log=False, precision=precision)
        lab1, C1, _, log = gkm.kmeans_fit(x, k, gi1, iters, init_labels=gkm.init_labels(n, k, fs), precision=precision)
        assert torch.equal(gi[first:first + n] - first, gi1) and torch.equal(gd[first:first + n], gd1)
        assert torch.equal(lab[first:first + n], lab1)
        assert torch.equal(C[kfirst:kfirst + k], C1)
        assert dist[j].item() == log[-1]
        first, kfirst = first + n, kfirst + k
