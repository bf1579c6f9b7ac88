"""The tensor-core screening of the recall estimator against its FP32 tiles: queries asked all at once are screened,
the same queries in small groups are not, and both give every query's exact nearest neighbour under the same key, bit
for bit."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n, d, m, kind, pad", [
    (20_000, 64, 800, "gauss", 0),     # two K-blocks of one, 3.1 query blocks
    (16_001, 128, 513, "int", 0),      # exact products, a last tile of one sample
    (40_003, 33, 777, "gauss", 0),     # rows that are not vectors
    (20_000, 70, 800, "gauss", 3),     # nor aligned ones
    (12_000, 192, 500, "gauss", 0),    # three K-blocks
    (9_000, 256, 500, "far", 0),       # four; samples far from the origin
    (5_000, 260, 800, "gauss", 0),     # five: the queries' operand is streamed
    (3_100, 960, 400, "gauss", 0),
    (7_000, 300, 500, "bf16", 0),
    (30_000, 96, 400, "same", 0),      # equal samples: every list overflows
    (20_000, 64, 800, "odd", 0),       # NaN, infinities, zeros, tiny and huge samples, ids out of range
])
def test_screened_equals_tiles(n, d, m, kind, pad):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1705_01813_gb300 import gkm
    assert n * d * m >= 1.0e9
    g = np.random.default_rng(n + d + m)
    c = max(4, n // 80)
    X = g.uniform(-10, 10, (c, d))[g.integers(0, c, n)] + g.standard_normal((n, d))
    if kind == "far":
        X += 3000.0
    if kind == "same":
        X[:] = X[0]
    X = X.astype(np.float32)
    if kind == "odd":
        X[5, 3], X[6, 1], X[7, 0] = np.nan, np.inf, -np.inf
        X[10:40] = 0.0
        X[50:60] *= 1e-24
        X[70:80] *= 1e18
        X[90:95] = X[90]
    t = torch.from_numpy(X).cuda()
    if kind == "int":
        t = (t * 6 + 64).round().clamp(0, 255)
    if kind == "bf16":
        t = t.to(torch.bfloat16)
    if pad:
        wide = torch.full((n, d + pad), 7.0, device="cuda")
        wide[:, :d] = t
        t = wide[:, :d]
    q = g.permutation(n)[:m].astype(np.int32)
    q[:100] = np.arange(100)  # the odd samples among the queries
    gi = g.integers(0, n, (n, 4)).astype(np.int32)
    if kind == "odd":
        gi[q[100:110], 0] = [-1, n, 2**31 - 1] * 3 + [-5]
        gi[q[110], 0] = q[110]
        q[m - 3:] = [n, -1, 2**31 - 1]
    gi, q = torch.from_numpy(gi).cuda(), torch.from_numpy(q).cuda()
    ws = gkm.Workspace(gkm.workspace_size(gkm.GK_OP_RECALL, n, d, m, 4))
    hits, nn, nd = gkm.graph_recall(t, gi, q, ws=ws)
    assert gkm.read_status(ws) == (gkm.GK_ERR_INVALID if kind == "odd" else gkm.GK_OK)
    step = int(0.99e9 / (n * d))
    total = 0
    for s in range(0, m, step):
        part = q[s:s + step].contiguous()
        h2, nn2, nd2 = gkm.graph_recall(t, gi, part, ws=ws)
        total += int(h2)
        assert torch.equal(nn[s:s + step], nn2)
        assert torch.equal(nd[s:s + step].view(torch.int32), nd2.view(torch.int32))
    assert int(hits) == total
