"""Int8 screening of samples and centroids of small magnitude, where products of the two rows' scales leave FP32's range:
labels and distances are those of the FP32 rows at every power of two."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("d", [32, 64, 128, 256, 512, 1024])
@pytest.mark.parametrize("exp", [0, -40, -56, -62, -64, -66, -68, -70])
def test_scaled_rows_keep_their_labels(d, exp):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1705_01813_gb300 import gkm
    n, k, kappa = 3001, 150, 24
    g = np.random.default_rng(d)
    X = g.uniform(-3, 3, (50, d))[g.integers(0, 50, n)] + g.standard_normal((n, d))
    X = torch.from_numpy(X.astype(np.float32)).cuda() * 2.0 ** exp
    X[11] = 0.0
    gi = torch.from_numpy(g.integers(0, n, (n, kappa)).astype(np.int32)).cuda()
    L = gkm.init_labels(n, k, 1)
    C = torch.zeros((k, d), device="cuda")
    gkm.update_step(X, L, k, C)
    C[:40] = X[:40]
    C[7], C[9] = C[8], 0.0
    for x in (X, X.to(torch.bfloat16)):
        want, best, s, _ = gkm.assign_step(x, gi, C, L, precision=0)
        got, b, s2, _ = gkm.assign_step(x, gi, C, L, precision=4)
        assert torch.equal(got, want), int((got != want).sum())
        assert torch.equal(b.view(torch.int32), best.view(torch.int32))
        assert float(s) == float(s2)


@pytest.mark.parametrize("d", [32, 64, 128, 256])
@pytest.mark.parametrize("exp", [-30, -34, -40, -60, -66, -70, -74])
def test_bf16_screenings_of_scaled_rows(d, exp):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1705_01813_gb300 import gkm
    n, k, kappa = 3001, 150, 24
    g = np.random.default_rng(d)
    X = g.uniform(-3, 3, (50, d))[g.integers(0, 50, n)] + g.standard_normal((n, d))
    X = torch.from_numpy(X.astype(np.float32)).cuda() * 2.0 ** exp
    gi = torch.from_numpy(g.integers(0, n, (n, kappa)).astype(np.int32)).cuda()
    L = gkm.init_labels(n, k, 1)
    C = torch.zeros((k, d), device="cuda")
    gkm.update_step(X, L, k, C)
    C[:100] = X[:100]
    C[100:] += X[:50] * 2.0 ** -7  # candidates that rounding decides
    off, mem, _ = gkm.group_by_label(L, k)
    want, best, s, _ = gkm.assign_step(X, gi, C, L, precision=0)
    for p in (2, 3):
        got, b, s2, _ = gkm.assign_step(X, gi, C, L, precision=p, members=mem)
        assert torch.equal(got, want), (p, int((got != want).sum()))
        assert torch.equal(b.view(torch.int32), best.view(torch.int32))


@pytest.mark.parametrize("d", [64, 100, 128])
@pytest.mark.parametrize("exp", [-40, -60, -64, -66, -68, -72])
def test_tensor_core_refinement_of_scaled_rows(d, exp):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1705_01813_gb300 import gkm
    n, k, kappa = 4001, 80, 20
    g = np.random.default_rng(d)
    X = g.uniform(-3, 3, (50, d))[g.integers(0, 50, n)] + 0.1 * g.standard_normal((n, d))
    X = torch.from_numpy(X.astype(np.float32)).cuda() * 2.0 ** exp
    L = gkm.init_labels(n, k, 2)
    for x in (X, X.to(torch.bfloat16)):
        gi, gd = gkm.init_graph(x, kappa, 5)
        gi2, gd2 = gi.clone(), gd.clone()
        gkm.graph_refine(x, L, k, gi, gd, precision=0)
        gkm.graph_refine(x, L, k, gi2, gd2, precision=1)
        assert torch.equal(gi, gi2), int((gi != gi2).sum())
        assert torch.equal(gd.view(torch.int32), gd2.view(torch.int32))
