"""The autotuner ranks the levels by whole fits (an iteration inside a fit costs less than an assignment by itself at the
levels that evaluate only what changed), and tries a group width only where the kernel reads it."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_1705_01813_gb300 import tune  # noqa: E402


def test_widths_only_where_the_kernel_reads_them():
    for p, d, want in [(0, 64, [0]), (0, 128, [8, 4]), (0, 512, [8, 4]), (0, 960, [0]), (1, 32, [0]), (1, 256, [8, 4]),
                       (1, 512, [0]), (2, 32, [8, 4]), (2, 512, [8, 4]), (2, 960, [0]), (3, 128, [0]), (4, 128, [0]),
                       (4, 960, [0])]:
        assert tune._widths(p, d) == want, (p, d)


@pytest.mark.gpu
def test_scores_follow_the_fits():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1705_01813_gb300 import gkm
    g = np.random.default_rng(3)
    n, d, k, tau, iters = 60_000, 96, 1200, 2, 6
    X = torch.from_numpy((g.uniform(-10, 10, (900, d))[g.integers(0, 900, n)]
                          + g.standard_normal((n, d))).astype(np.float32)).cuda()
    gi, gd, _, _ = gkm.build_knn_graph(X, 16, xi=50, tau=tau, seed=1)
    lab, C, cnt, _ = gkm.kmeans_fit(X, k, gi, iters, seed=1)
    gi0, gd0, lab0 = gi.clone(), gd.clone(), lab.clone()
    r = tune.tune_precision(X, gi, gd, lab, k, tau=tau, iters=iters, use_cache=False)
    assert torch.equal(gi, gi0) and torch.equal(gd, gd0) and torch.equal(lab, lab0)
    assert set(r["fit_ms"]) == {0, 1, 2, 3, 4} and min(r["fit_ms"].values()) > 0
    refine = r["refine_ms"]["fp32_tiles"] - r["refine_ms"]["precision_ge_1"]
    for p in range(1, 5):  # the copies' time is the same in all scores
        diff = (r["fit_ms"][p] - r["fit_ms"][0]) / iters * (tau + iters) - refine * tau
        assert abs(r["score_ms"][p] - r["score_ms"][0] - diff) < 1e-6 * max(r["score_ms"].values())
    assert r["group_width_by_level"][3] == r["group_width_by_level"][4] == 0
    assert r["group_width_by_level"][0] in (4, 8)
