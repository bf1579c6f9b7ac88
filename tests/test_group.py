"""Grouping by label at the edges of its passes, tiles and blocks, against numpy's stable sort (bit-exact)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n, k, kind", [
    (1, 1, "uniform"),
    (31, 2, "uniform"),
    (2048, 1023, "uniform"),        # one pass, one whole tile
    (2049, 1024, "uniform"),        # two passes, a second tile of one element
    (1216 * 2048, 900, "uniform"),  # every block one tile
    (1216 * 2048 + 1, 70000, "uniform"),  # blocks of two tiles, some without any
    (200_001, 1 << 20, "uniform"),  # three passes, mostly empty clusters
    (100_003, 5000, "one"),         # everything in one cluster
    (100_003, 5000, "sorted"),
    (50_001, 300, "invalid"),       # labels out of range: in no cluster, after every valid one
    (50_001, 3000, "invalid"),
])
def test_group_equals_stable_sort(n, k, kind):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1705_01813_gb300 import gkm
    g = np.random.default_rng(n + k)
    L = g.integers(0, k, n).astype(np.int32)
    if kind == "one":
        L[:] = k // 2
    elif kind == "sorted":
        L.sort()
    elif kind == "invalid":
        L[g.integers(0, n, 700)] = np.array([-1, k, 2**31 - 1, -(2**31)], np.int32)[g.integers(0, 4, 700)]
    valid = (L >= 0) & (L < k)
    ws = gkm.Workspace(gkm.workspace_size(gkm.GK_OP_UPDATE, n, 1, k))
    off, mem, cnt = gkm.group_by_label(torch.from_numpy(L).cuda(), k, ws=ws)
    assert gkm.read_status(ws) == (gkm.GK_OK if valid.all() else gkm.GK_ERR_INVALID)
    key = np.where(valid, L.astype(np.int64), k)
    counts = np.bincount(key, minlength=k + 1)[:k]
    assert np.array_equal(mem.cpu().numpy(), np.argsort(key, kind="stable"))
    assert np.array_equal(cnt.cpu().numpy(), counts)
    assert np.array_equal(off.cpu().numpy(), np.concatenate([[0], np.cumsum(counts)]))
