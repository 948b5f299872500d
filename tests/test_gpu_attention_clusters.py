"""Small launches of the fp32 kernel, whose splits a cluster merges by itself: one to eight splits, both head dimensions, ratios that
leave a last row block short, sequences that end in every split, trees of one row and of all.  Tolerance: that of the
splits (fp32 sums over at most 200 keys)."""
import pytest

from test_gpu_attention_splits import _compare

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("Hq,Hkv,d", [(1, 1, 64), (2, 1, 128), (3, 1, 64), (5, 1, 128)])
@pytest.mark.parametrize("plens,P", [([0], 0), ([40, 0, 7], 40), ([136, 31], 136), ([190], 190), ([100], 190)])
@pytest.mark.parametrize("M", [1, 30, 64])
def test_splits_merged_by_a_cluster(Hq, Hkv, d, plens, P, M):
    _compare(len(plens), Hq, Hkv, d, plens, P, M)
