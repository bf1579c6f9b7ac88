"""Every precision level gives the FP32 assignment's labels and distances bit for bit, at the widths where the screening's
row formats change (384, 640, 768 and 896 read the int8 shadow in the wrong order once)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dtype", ["f32", "bf16"])
@pytest.mark.parametrize("d", [32, 36, 60, 64, 68, 128, 132, 256, 260, 384, 512, 516, 640, 768, 896, 1020, 1024])
def test_screened_labels_equal_fp32(d, dtype):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1705_01813_gb300 import gkm
    n, k, kappa = 6001, 240, 33
    g = np.random.default_rng(d)
    X = g.uniform(0, 1, (60, d))[g.integers(0, 60, n)] + 0.3 * g.standard_normal((n, d))
    X = torch.from_numpy(X.astype(np.float32)).cuda()
    if dtype == "bf16":
        X = X.to(torch.bfloat16)
    gi = torch.from_numpy(g.integers(0, n, (n, kappa)).astype(np.int32)).cuda()
    L = gkm.init_labels(n, k, 1)
    C = torch.zeros((k, d), device="cuda")
    gkm.update_step(X, L, k, C)
    C[:40] *= 1.0 + torch.linspace(-0.5, 0.5, 40, device="cuda")[:, None]  # candidates that are told apart
    C[7], C[9] = C[8], 0.0
    want, best, s, _ = gkm.assign_step(X, gi, C, L, precision=0)
    for p in (1, 2, 4, 4 | (4 << 8), 4 | (8 << 8)):
        got, b, s2, _ = gkm.assign_step(X, gi, C, L, precision=p)
        assert torch.equal(got, want), p
        assert torch.equal(b.view(torch.int32), best.view(torch.int32)), p
        assert float(s2) == float(s)


@pytest.mark.parametrize("kappa", [1, 20, 31, 32, 50, 128])
@pytest.mark.parametrize("d", [4, 12, 28, 32, 36, 56, 64])
def test_narrow_rows_equal_zero_padded_rows(d, kappa):
    # rows of at most 64 values take several candidates to a load; zero columns up to 68 values change no distance's bits
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1705_01813_gb300 import gkm
    n, k = 5003, 150
    g = np.random.default_rng(d * 131 + kappa)
    gi = torch.from_numpy(g.integers(0, n, (n, kappa)).astype(np.int32)).cuda()
    L = torch.from_numpy(g.integers(0, k, n).astype(np.int32)).cuda()
    for bf16 in (False, True):
        X = torch.from_numpy(g.standard_normal((n, d)).astype(np.float32)).cuda()
        C = torch.from_numpy(g.standard_normal((k, d)).astype(np.float32)).cuda()
        C[5] = C[6]  # equal distances
        Xw, Cw = torch.zeros((n, 68), device="cuda"), torch.zeros((k, 68), device="cuda")
        Xw[:, :d], Cw[:, :d] = X, C
        if bf16:
            X, Xw = X.to(torch.bfloat16), Xw.to(torch.bfloat16)
        got, b, s, _ = gkm.assign_step(X, gi, C, L, precision=1)
        want, bw, sw, _ = gkm.assign_step(Xw, gi, Cw, L, precision=1)
        assert torch.equal(got, want)
        assert torch.equal(b.view(torch.int32), bw.view(torch.int32))
        assert float(s) == float(sw)
