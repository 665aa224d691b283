"""The quality metrics' workspace holds what the kernels use: the overlaps and
four 8-byte arrays per superpixel (perimeter, largest overlap, undersegmentation,
compactness), two counts and four results, each on a 256-byte boundary."""
import pytest

from paper_1903_07149_gb300 import build as scalp_build
from paper_1903_07149_gb300 import scalp


@pytest.fixture(scope="module", autouse=True)
def built():
    scalp_build.build()


@pytest.mark.parametrize("n_labels,n_gt", [(1, 1), (64, 7), (2000, 300), (10001, 40), (1 << 20, 256)])
def test_workspace_is_what_is_used(n_labels, n_gt):
    up = lambda v: (v + 255) & ~255
    want = up(4 * n_labels * n_gt) + 4 * up(8 * n_labels) + up(16) + up(32)
    assert scalp.scalp_quality_workspace_bytes(100, 100, n_labels, n_gt) == want
