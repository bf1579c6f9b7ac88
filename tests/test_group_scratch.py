"""The grouping's part of a workspace holds its four key and value buffers, each aligned by itself (sized as one buffer they
were up to 768 bytes short and reached past the grouping's scratch)."""
import pytest

pytest.importorskip("torch")

from paper_1705_01813_gb300 import gkm  # noqa: E402


def _al(b):
    return (b + 255) // 256 * 256


@pytest.mark.parametrize("n", [2, 63, 64, 65, 1_000, 2_049, 300_000, 300_007, 2_500_000])
@pytest.mark.parametrize("k", [1, 200, 1_023, 1_024])
def test_workspace_holds_the_groupings_buffers(n, k):
    if k > n:
        pytest.skip("more clusters than samples")
    csr = _al(4 * (k + 1)) + _al(4 * n) + _al(4 * k)  # offsets, members, counts
    tiles = (n + 2047) // 2048
    scratch = 4 * _al(4 * n) + _al(4 * 1024 * min(tiles, 1216)) + 4 * 1024  # buffers, blocks' digit counts, totals
    assert gkm.workspace_size(gkm.GK_OP_BOOST, n, 8, k) >= csr + scratch
