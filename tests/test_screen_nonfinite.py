"""Screened assignments of samples and centroids with NaN or infinity: every level gives level 0's labels and distances."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("kappa", [3, 40])
@pytest.mark.parametrize("d", [32, 72, 128, 256, 512, 960])
def test_levels_agree(d, kappa):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1705_01813_gb300 import gkm
    n, k = 3001, 120
    g = np.random.default_rng(d + kappa)
    X = g.uniform(-3, 3, (50, d))[g.integers(0, 50, n)] + g.standard_normal((n, d))
    X[5, 1], X[6, 0], X[7, 3], X[8] = np.nan, np.inf, -np.inf, np.inf
    X = torch.from_numpy(X.astype(np.float32)).cuda()
    gi = torch.from_numpy(g.integers(0, n, (n, kappa)).astype(np.int32)).cuda()
    L = torch.from_numpy(g.integers(0, k, n).astype(np.int32)).cuda()
    C = torch.from_numpy(g.standard_normal((k, d)).astype(np.float32)).cuda()
    C[3, 2], C[4, 0], C[5] = float("nan"), float("inf"), float("-inf")
    L[20:60], gi[20:60] = 4, torch.arange(20, 60, device="cuda", dtype=torch.int32)[:, None]  # no finite candidate
    _, mem, _ = gkm.group_by_label(L, k)
    for x in (X, X.to(torch.bfloat16)):
        want, best, s, _ = gkm.assign_step(x, gi, C, L, precision=0)
        for p in (1, 2, 4) + ((3,) if x.dtype == torch.float32 else ()):
            got, b, _, _ = gkm.assign_step(x, gi, C, L, precision=p, members=mem)
            assert torch.equal(got, want), (p, torch.nonzero(got != want)[:5, 0].tolist())
            assert torch.equal(b.view(torch.int32), best.view(torch.int32)), p
    gkm.read_status(gkm.workspace(1))
