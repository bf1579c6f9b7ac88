"""The centroid update's block kernel: rows of several column blocks, and its two ways through the clusters (a block each,
or a walk over chunks where most clusters are small), against FP64 means of the same groups."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("sizes", ["even", "one_large", "many_small"])
@pytest.mark.parametrize("d", [4, 128, 129, 132, 256, 384, 500, 512, 516, 640, 1024, 1028, 1100])
def test_update_of_split_rows(d, sizes):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1705_01813_gb300 import gkm
    g = np.random.default_rng(d)
    if sizes == "even":
        k, n = 7, 1501
        L = g.integers(0, k - 1, n)  # the last cluster is empty
    elif sizes == "one_large":
        k, n = 30, 5000
        L = np.where(g.random(n) < 0.8, 3, g.integers(0, k, n))
    else:
        k, n = 3000, 9000
        L = np.where(g.random(n) < 0.1, g.integers(0, 3, n) * 997, g.integers(0, k, n))
    L = torch.from_numpy(L.astype(np.int32)).cuda()
    X = torch.from_numpy(g.standard_normal((n, d)).astype(np.float32)).cuda()
    outs = []
    for Xt in (X, X.to(torch.bfloat16), X.to(torch.bfloat16).float()):
        C = torch.full((k, d), 7.0, device="cuda")
        r = gkm.update_step(Xt, L, k, C)
        cnt = torch.bincount(L.long(), minlength=k)
        want = torch.zeros((k, d), dtype=torch.float64, device="cuda").index_add_(0, L.long(), Xt.double())
        mean = want / cnt.clamp(min=1)[:, None]
        full = cnt > 0
        # one FP32 rounding of a mean below 8 (2^-22), the compensated sum's error far below it
        assert float((C.double() - mean)[full].abs().max()) <= 2.0 ** -22
        d2 = (Xt.double().square().sum() - (want.square().sum(1)[full] / cnt[full]).sum())
        s = [t for t in (r if isinstance(r, tuple) else (r,)) if torch.is_tensor(t) and t.dtype == torch.float64]
        for t in s:
            assert abs(float(t.flatten()[0]) - float(d2)) <= 1e-6 * float(Xt.double().square().sum())
        outs.append((C, s))
    assert torch.equal(outs[1][0], outs[2][0])  # BF16 samples sum as their FP32 widening
    assert all(torch.equal(a, b) for a, b in zip(outs[1][1], outs[2][1]))
