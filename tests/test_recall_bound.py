"""The recall estimator's screening bound on FP32 samples that BF16 rounds by close to its unit, 2^-8 of a value: rows
whose distances are small beside their norms.  With the true neighbour in the graph, every query asked at once must give
the key that the FP32 tiles give it (the same queries in groups too small to be screened)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu


def _check(X, q, gi, name_truth):
    """X, q, gi on the device; name_truth: the graph rows of the queries start with the true neighbour."""
    from paper_1705_01813_gb300 import gkm
    (n, d), m = X.shape, q.numel()
    assert n * d * m >= 1.0e9  # screened when asked at once
    step = int(0.99e9 / (n * d))
    parts = [gkm.graph_recall(X, gi, q[s:s + step].contiguous()) for s in range(0, m, step)]
    nn, nd = torch.cat([p[1] for p in parts]), torch.cat([p[2] for p in parts])
    if name_truth:
        gi[q.long(), 0] = nn
    hits, nn2, nd2 = gkm.graph_recall(X, gi, q)
    wrong = int((nn != nn2).sum())
    assert wrong == 0, f"{wrong} of {m} queries have another neighbour"
    assert torch.equal(nd.view(torch.int32), nd2.view(torch.int32))
    assert not name_truth or int(hits) == m


def test_sample_at_the_rounding_unit():
    # query b (entries 1 and 2, which BF16 holds), its neighbour (1 + 2^-8) b, which BF16 rounds to b, and a sample that
    # BF16 holds at 20 times the distance, named by the graph
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    d, m, n = 128, 400, 20_000
    g = np.random.default_rng(1)
    X = g.integers(1, 3, (n, d)).astype(np.float32)
    X[m:2 * m] = X[:m] * np.float32(1 + 2.0 ** -8)
    X[2 * m:3 * m] = X[:m]
    X[2 * m:3 * m, 0] += 0.3125
    gi = np.tile(np.arange(n, dtype=np.int32)[::-1, None], (1, 2)).copy()
    gi[:m] = np.arange(2 * m, 3 * m, dtype=np.int32)[:, None]
    t, gi = torch.from_numpy(X).cuda(), torch.from_numpy(gi).cuda()
    q = torch.arange(m, dtype=torch.int32, device="cuda")
    _check(t, q, gi, False)
    from paper_1705_01813_gb300 import gkm
    _, nn, _ = gkm.graph_recall(t, gi, q)
    assert torch.equal(nn, q + m)


@pytest.mark.parametrize("n, d, m, kind", [
    (400_000, 2, 1300, "gauss"),
    (300_000, 3, 1200, "gauss"),
    (200_000, 4, 1300, "gauss"),
    (60_000, 16, 1100, "gauss"),
    (40_000, 32, 900, "column"),      # one column scaled by 1,000 carries the norm
    (12_000, 128, 800, "column"),
    (7_000, 200, 800, "column"),      # the queries' operand is streamed
    (40_000, 32, 900, "lognormal"),
    (30_000, 33, 1100, "lognormal"),  # rows that are not vectors
])
def test_screened_equals_tiles_where_rounding_is_large(n, d, m, kind):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    g = np.random.default_rng(n + d)
    X = g.standard_normal((n, d))
    if kind == "column":
        X[:, d // 2] *= 1000.0
    if kind == "lognormal":
        X = np.exp(2.0 * X)
    q = torch.from_numpy(g.permutation(n)[:m].astype(np.int32)).cuda()
    gi = torch.from_numpy(g.integers(0, n, (n, 3)).astype(np.int32)).cuda()
    _check(torch.from_numpy(X.astype(np.float32)).cuda(), q, gi, True)
