"""A fit evaluates only what the previous iteration's moves can have changed (candidates of changed clusters; sums of
changed clusters).  Labels, centroids, sizes and the distortion log must be those of the same iterations driven step by
step, where every assignment evaluates all candidates and every update all clusters, bit for bit."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n, d, k, kappa, dtype, precision, spoil", [
    (4001, 32, 40, 20, "f32", 0, None),        # too small to be tracked
    (131072, 32, 400, 20, "f32", 0, None),     # the smallest size that is; few clusters
    (131071, 32, 13000, 20, "f32", 1, None),   # one sample less, many small clusters
    (131073, 33, 1000, 16, "f32", 0, None),    # rows that are not 16-byte vectors
    (4001, 1100, 80, 16, "f32", 0, None),      # rows wider than the row kernels take
    (33001, 128, 3000, 50, "int", 2, None),    # BF16 screening; equal distances
    (8501, 512, 800, 40, "bf16", 4 | (4 << 8), None),
    (14101, 300, 700, 128, "f32", 4, None),    # int8 rows that are not lane-major, the largest kappa
    (66001, 64, 66001, 8, "f32", 1, None),     # as many clusters as samples
    (90001, 48, 1000, 33, "f32", 1, "nan"),    # a non-finite sample in one cluster
    (90001, 48, 1000, 16, "f32", 4, "inf"),
    (45001, 96, 500, 16, "int", 3, None),      # precision 3 keeps nothing between iterations
])
def test_fit_equals_full_iterations(n, d, k, kappa, dtype, precision, spoil):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1705_01813_gb300 import gkm
    g = np.random.default_rng(n + d + k)
    c = max(4, min(k, n // 8))
    X = g.uniform(-4, 4, (c, d))[g.integers(0, c, n)] + g.standard_normal((n, d))
    X = torch.from_numpy(X.astype(np.float32)).cuda()
    if dtype == "int":
        X = (X * 8 + 40).round().clamp(0, 255)
    if dtype == "bf16":
        X = X.to(torch.bfloat16)
    if spoil:
        X[17, 3] = float(spoil)
    gi, _, _, _ = gkm.build_knn_graph(X, kappa, tau=3, seed=1, precision=min(precision & 255, 1))
    L = gkm.init_labels(n, k, 9)
    iters = 12
    lab, C, cnt, log = gkm.kmeans_fit(X, k, gi, iters, init_labels=L, precision=precision)
    ref = torch.zeros((k, d), device="cuda")
    _, cnt2, e, _, _ = gkm.update_step(X, L, k, ref)
    want = [float(e) / n]
    for _ in range(iters):
        L, _, s, _ = gkm.assign_step(X, gi, ref, L, precision=precision)
        want.append(float(s) / n)
        _, cnt2, e, _, _ = gkm.update_step(X, L, k, ref)
        want.append(float(e) / n)
    status = gkm.read_status(gkm.workspace(1))  # the calls above share this thread's workspace; read and cleared
    assert status == (gkm.GK_ERR_NUMERIC if spoil else gkm.GK_OK)
    assert torch.equal(lab, L) and torch.equal(cnt, cnt2)
    assert torch.equal(C.view(torch.int32), ref.view(torch.int32))
    assert np.array_equal(np.array(log), np.array(want), equal_nan=True)
