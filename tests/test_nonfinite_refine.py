"""The tensor-core refinement on samples with NaN or infinity: the graph is that of the FP32 tiles, in a single call (also
for runs whose first member, on which FP32 runs are centred, is such a sample, and for rows that hold one), and within a
construction, where a pair that was left out would not be offered again."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu


def _samples(n, d, kind, dtype, seed):
    g = np.random.default_rng(seed)
    X = g.uniform(-10, 10, (max(2, n // 60), d))[g.integers(0, max(2, n // 60), n)] + g.standard_normal((n, d))
    if kind.startswith("int"):
        X = np.rint(X * 6 + 64).clip(0, 255)
    X = X.astype(np.float32)
    for i, v in ((0, np.nan), (n // 3, np.inf), (n // 2, -np.inf), (n - 1, np.nan)):
        X[i, i % d] = v
    if kind.endswith("rows"):
        X[n // 5] = np.nan
    X = torch.from_numpy(X).cuda()
    return X.to(torch.bfloat16) if dtype == "bf16" else X


CASES = [(3_001, 64, 12), (4_003, 72, 33), (5_000, 100, 70), (2_500, 128, 50)]


@pytest.mark.parametrize("dtype", ["f32", "bf16"])
@pytest.mark.parametrize("kind", ["gauss", "int", "int rows"])
@pytest.mark.parametrize("n, d, kappa", CASES)
def test_call_equals_fp32_tiles(n, d, kappa, kind, dtype):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1705_01813_gb300 import gkm
    X = _samples(n, d, kind, dtype, n + d)
    gi, gd = gkm.init_graph(X, kappa, 5)
    a, b = (gi.clone(), gd.clone()), (gi.clone(), gd.clone())
    for seed in (7, 8):
        L = gkm.init_labels(n, max(1, n // 50), seed)
        gkm.graph_refine(X, L, max(1, n // 50), *a, precision=0)
        gkm.graph_refine(X, L, max(1, n // 50), *b, precision=1)
        assert torch.equal(a[0], b[0])
        assert torch.equal(a[1].view(torch.int32), b[1].view(torch.int32))
    gkm.read_status(gkm.workspace(1))


@pytest.mark.parametrize("dtype", ["f32", "bf16"])
@pytest.mark.parametrize("n, d, kappa", CASES + [(45_001, 96, 10), (33_001, 128, 50)])
def test_construction_equals_level_0(n, d, kappa, dtype):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1705_01813_gb300 import gkm
    X = _samples(n, d, "gauss", dtype, n + d)
    a, b = (gkm.build_knn_graph(X, kappa, xi=30, tau=6, seed=5, want_log=False, precision=p) for p in (0, 1))
    gkm.read_status(gkm.workspace(1))
    assert torch.equal(a[2], b[2]) and torch.equal(a[0], b[0])
    assert torch.equal(a[1].view(torch.int32), b[1].view(torch.int32))
