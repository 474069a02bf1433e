"""The column pass ranks a warp's instances by column through one shared word per column.  From one
column (every lane in the same word) to the 255 the pass allows, over rounds that end inside a
warp and rows of several rounds, the lists are those of the KEY64 schedule, bit for bit."""
import numpy as np
import pytest

from test_gpu_binning import _screen
from test_gpu_binning_sizes import _binned

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("W,H,n,rmax", [(16, 16, 9001, 8), (7, 400, 20_000, 30), (33, 48, 9001, 60),
                                        (128, 20, 12_345, 5), (4080, 40, 30_000, 300), (4079, 700, 9001, 20)])
def test_lists_from_one_column_to_the_most(W, H, n, rmax):
    sp = _screen(170 + W, n, W, H, rmax, culled=0.1, ties=0.2, huge=3)
    a, b = (_binned(sp, W, H, mode, 6_000_000) for mode in ("two_phase", "key64"))
    assert a[0] == b[0] and a[1] == b[1]
    for x, y in zip(a[2:], b[2:]):
        assert np.array_equal(x, y)
