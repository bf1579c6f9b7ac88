"""Precision 0 is FP32 throughout: whatever the sizes, its assignment reads the FP32 centroid rows and screens nothing, so
that it stands as the reference of the other levels, in single calls and within a fit."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu

SIZES = [(10_923, 384, 300, 20), (6_001, 768, 240, 33), (4_100, 1024, 4_100, 9), (14_000, 300, 40, 1)]  # n d >= 2^22


def _case(n, d, k, kappa, dtype):
    from paper_1705_01813_gb300 import gkm
    g = np.random.default_rng(d)
    X = g.uniform(0, 1, (60, d))[g.integers(0, 60, n)] + 0.3 * g.standard_normal((n, d))
    X = torch.from_numpy(X.astype(np.float32)).cuda()
    X = X.to(torch.bfloat16) if dtype == "bf16" else X
    gi = torch.from_numpy(g.integers(0, n, (n, kappa)).astype(np.int32)).cuda()
    return X, gi, gkm.init_labels(n, k, 1)


def _kernels(call):
    from torch.profiler import ProfilerActivity, profile
    for _ in range(2):  # a first profiling session may come back empty while the profiler initialises
        with profile(activities=[ProfilerActivity.CUDA]) as prof:
            call()
            torch.cuda.synchronize()
        names = [e.name for e in prof.events() if e.device_type.name == "CUDA" and "gkm::" in e.name]
        if names:
            return names
    pytest.skip("the profiler recorded no kernel names here")


@pytest.mark.parametrize("dtype", ["f32", "bf16"])
@pytest.mark.parametrize("n, d, k, kappa", SIZES)
def test_level_0_screens_nothing(n, d, k, kappa, dtype):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1705_01813_gb300 import gkm
    assert n * d >= 1 << 22
    X, gi, L = _case(n, d, k, kappa, dtype)
    C = torch.zeros((k, d), device="cuda")
    gkm.update_step(X, L, k, C)
    for call in (lambda: gkm.assign_step(X, gi, C, L, precision=0),
                 lambda: gkm.kmeans_fit(X, k, gi, 3, init_labels=L, precision=0)):
        names = _kernels(call)
        assert any("k_assign_rows<" in nm for nm in names)
        assert not [nm for nm in names if "k_assign_rows_scr" in nm or "k_shadow" in nm]
    want, best, s, _ = gkm.assign_step(X, gi, C, L, precision=0)
    for p in (1, 2, 4):
        got, b, s2, _ = gkm.assign_step(X, gi, C, L, precision=p)
        assert torch.equal(got, want), p
        assert torch.equal(b.view(torch.int32), best.view(torch.int32)), p
        assert float(s2) == float(s)


@pytest.mark.parametrize("dtype", ["f32", "bf16"])
@pytest.mark.parametrize("n, d, k, kappa", SIZES)
def test_levels_of_a_fit_agree(n, d, k, kappa, dtype):
    # the lists of samples that may have changed, on FP32 rows and screened
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1705_01813_gb300 import gkm
    X, gi, L = _case(n, d, k, kappa, dtype)
    want = gkm.kmeans_fit(X, k, gi, 6, init_labels=L, precision=0)
    ref, lab = torch.zeros((k, d), device="cuda"), L
    gkm.update_step(X, lab, k, ref)
    for _ in range(6):
        lab, _, _, _ = gkm.assign_step(X, gi, ref, lab, precision=0)
        gkm.update_step(X, lab, k, ref)
    assert torch.equal(want[0], lab) and torch.equal(want[1].view(torch.int32), ref.view(torch.int32))
    for p in (1, 2, 4):
        got = gkm.kmeans_fit(X, k, gi, 6, init_labels=L, precision=p)
        assert torch.equal(got[0], want[0]), p
        assert torch.equal(got[1].view(torch.int32), want[1].view(torch.int32)), p
        assert got[3] == want[3]
