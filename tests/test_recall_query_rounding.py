"""The recall screening's bound takes the queries' own rounding errors in BF16.  A query at the rounding unit, whose
neighbour and decoy BF16 holds: the key must be that of the FP32 tiles; a bound that counts the query's error for 6% less
than it is loses the neighbour."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")


@pytest.mark.gpu
@pytest.mark.parametrize("d, scale", [(128, 1.0), (200, 1.0), (99, 2.0 ** -20)])
def test_query_at_the_rounding_unit(d, scale):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1705_01813_gb300 import gkm
    n, m = 42_000, 256
    g = np.random.default_rng(d)
    X = g.standard_normal((n, d)).astype(np.float32)
    X[1:m:2] = -X[0:m:2]  # the queries in pairs x, -x: their mean, the centre, is zero
    X[0], X[1] = 1 + 2.0 ** -8, -(1 + 2.0 ** -8)  # BF16 rounds to 1 and -1
    X[m], X[m + 1] = 1 + 2.0 ** -7, -(1 + 2.0 ** -7)  # their neighbours
    X[m + 2], X[m + 3] = 1 - 2.0 ** -6, -(1 - 2.0 ** -6)  # what the graph names
    gi = g.integers(m + 4, n, (n, 3)).astype(np.int32)
    gi[0, 0], gi[1, 0] = m + 2, m + 3
    X, gi = torch.from_numpy(X * np.float32(scale)).cuda(), torch.from_numpy(gi).cuda()
    q = torch.arange(m, dtype=torch.int32, device="cuda")
    assert n * d * m >= 1.0e9
    step = int(0.99e9 / (n * d))  # groups that the tiles take
    parts = [gkm.graph_recall(X, gi, q[s:s + step].contiguous()) for s in range(0, m, step)]
    _, nn, nd = gkm.graph_recall(X, gi, q)
    assert nn[:2].tolist() == [m, m + 1]
    assert torch.equal(nn, torch.cat([p[1] for p in parts]))
    assert torch.equal(nd.view(torch.int32), torch.cat([p[2] for p in parts]).view(torch.int32))
