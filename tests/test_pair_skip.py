"""Graph construction compares a pair once: rounds after the first leave out the pairs that shared a run in the round
before.  The graph must be that of the same rounds driven step by step, where every refinement compares all pairs of
its runs, bit for bit."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu


def _samples(n, d, kind, seed):
    g = np.random.default_rng(seed)
    X = g.uniform(-10, 10, (max(4, n // 60), d))[g.integers(0, max(4, n // 60), n)] + g.standard_normal((n, d))
    X = torch.from_numpy(X.astype(np.float32)).cuda()
    if kind == "int":
        X = (X * 6 + 64).round().clamp(0, 255)
    return X.to(torch.bfloat16) if kind == "bf16" else X


@pytest.mark.parametrize("n, d, kind, kappa, max_cluster, precision", [
    (4099, 33, "f32", 20, 128, 0),     # FP32 tiles, element loads, odd width
    (4099, 32, "f32", 50, 64, 0),      # no long runs
    (3001, 300, "f32", 32, 128, 1),    # wide FP32 rows
    (4099, 512, "bf16", 40, 128, 1),   # the warp-specialised kernel
    (3001, 100, "bf16", 33, 128, 0),   # BF16 rows not a multiple of 16 bytes
    (5003, 128, "int", 50, 128, 1),    # tensor cores, exact Gram
    (5003, 100, "f32", 65, 128, 1),    # tensor cores, recomputed pairs, three row slots
    (4099, 64, "f32", 128, 300, 1),    # runs longer than a tile, the largest kappa
    (4099, 48, "f32", 1, 200, 0),      # one neighbour, several tiles per run
    (1000, 16, "f32", 10, 2, 0),       # runs of two and single left-over members
    (70, 8, "f32", 69, 128, 0),        # one cluster: everything is compared in the first round
])
def test_one_call_equals_rounds_that_compare_everything(n, d, kind, kappa, max_cluster, precision):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1705_01813_gb300 import gkm
    X = _samples(n, d, kind, n + d)
    xi, tau = 50, 6
    k0 = max(1, n // xi)
    gi, gd, lab, _ = gkm.build_knn_graph(X, kappa, xi=xi, tau=tau, max_cluster=max_cluster, seed=5, precision=precision)
    gi2, gd2 = gkm.init_graph(X, kappa, 5)
    L = gkm.init_labels(n, k0, 5)
    C = torch.zeros((k0, d), device="cuda")
    gkm.update_step(X, L, k0, C)
    for _ in range(tau):
        L, _, _, _ = gkm.assign_step(X, gi2, C, L, precision=precision)
        gkm.update_step(X, L, k0, C)
        gkm.graph_refine(X, L, k0, gi2, gd2, max_cluster=max_cluster, precision=precision)
    assert torch.equal(lab, L)
    assert torch.equal(gi, gi2)
    assert torch.equal(gd.view(torch.int32), gd2.view(torch.int32))
