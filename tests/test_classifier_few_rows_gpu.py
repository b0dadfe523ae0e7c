"""The fused classifier for few rows at the edges of its tiles: one row, counts around the three tile widths, features
that fill no K-block and more than one ring, shards of less than a chunk and of an odd number of chunks, labels on
a shard's first and last class, and that wide features and many rows still take the other kernel.  Oracle and
tolerances as for the fused classifier elsewhere."""
import pytest

from test_ops_gpu import _fused_classifier_case

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("rows", [1, 31, 32, 33, 64, 65, 127, 128, 129])
@pytest.mark.parametrize("feat,classes,k", [(8, 64, 8), (72, 4960, 4), (512, 2 * 136, 2), (200, 3 * 392, 3)])
def test_few_rows(rows, feat, classes, k):
    _fused_classifier_case(rows, feat, classes, k, seed=3100 + rows)


@pytest.mark.parametrize("rows,feat,classes,k", [(32, 2048, 520, 1), (100, 2000, 1040, 2), (16, 64, 148 * 256 * 3 + 40, 1)])
def test_wide_features_and_several_tiles_a_pair(rows, feat, classes, k):
    _fused_classifier_case(rows, feat, classes, k, seed=3200)
