"""The binned likelihood path with tiles of 64 anchors (large frames): particle
counts around one and two work items of 2560 records, all in one tile, at the
largest window (radius 8), the smallest (0) and the usual one.  The direct path
is the reference, bit for bit."""
import pytest
from test_gpu_binned_items import _compare

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("radius", [0, 5, 8])
@pytest.mark.parametrize("n", [1, 511, 2559, 2560, 2561, 5120, 5123])
def test_binned_equals_direct_in_one_wide_tile(n, radius):
    _compare(n, False, 1800, 1900, radius)


def test_binned_equals_direct_at_the_most_bins():
    # 55 x 55 tiles of 64 anchors, close to the 3073 bins a context may have
    _compare(60_001, True, 3500, 3500, 8)
