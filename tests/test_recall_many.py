"""Recall over many queries: the screening takes them in batches, so that its lists have a bounded size however many
there are, and every query gets the key that the FP32 tiles give it."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")


@pytest.mark.parametrize("n, d", [(1_000_000, 128), (100_000, 960)])
def test_workspace_is_bounded(n, d):
    # all samples as queries: a few words a query beside a fixed part
    from paper_1705_01813_gb300 import gkm
    small, large = (gkm.workspace_size(gkm.GK_OP_RECALL, n, d, m, 10) for m in (n // 10, n))
    assert large - small <= 16 * n
    assert large <= 16 * n + (256 << 20)


@pytest.mark.gpu
@pytest.mark.parametrize("n, d, m, kind", [
    (1_500, 96, 9_728, "gauss"),        # a full batch
    (1_500, 96, 9_729, "gauss"),        # and one query more
    (2_000, 64, 2 * 9_728 + 300, "gauss"),
    (1_200, 132, 30_001, "int"),
    (1_001, 40, 30_000, "same"),        # equal samples: every list overflows and goes to the tiles
])
def test_batches_equal_tiles(n, d, m, kind):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1705_01813_gb300 import gkm
    assert n * d * m >= 1.0e9
    g = np.random.default_rng(m)
    X = g.uniform(-10, 10, (40, d))[g.integers(0, 40, n)] + g.standard_normal((n, d))
    if kind == "int":
        X = np.rint(X * 6 + 64)
    if kind == "same":
        X[:] = X[0]
    X = torch.from_numpy(X.astype(np.float32)).cuda()
    q = g.integers(0, n, m).astype(np.int32)
    q[[0, m // 2, m - 1]] = [-1, n, 2**31 - 1]  # no samples: never hits
    gi = torch.from_numpy(g.integers(0, n, (n, 5)).astype(np.int32)).cuda()
    q = torch.from_numpy(q).cuda()
    ws = gkm.Workspace(gkm.workspace_size(gkm.GK_OP_RECALL, n, d, m, 5))
    hits, nn, nd = gkm.graph_recall(X, gi, q, ws=ws)
    assert gkm.read_status(ws) == gkm.GK_ERR_INVALID
    step, total = int(0.99e9 / (n * d)), 0
    for s in range(0, m, step):
        h2, nn2, nd2 = gkm.graph_recall(X, gi, q[s:s + step].contiguous())
        total += int(h2)
        assert torch.equal(nn[s:s + step], nn2)
        assert torch.equal(nd[s:s + step].view(torch.int32), nd2.view(torch.int32))
    gkm.read_status(gkm.workspace(1))  # the groups' calls noted the ids out of range
    assert int(hits) == total
