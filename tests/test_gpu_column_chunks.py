"""The column passes take 256, 512, 1,024 or 2,048 row-sorted records per chunk, by the number of
records of the launch: with each size the lists, ranges and render order are those of the KEY64
schedule, which has no column pass."""
import numpy as np
import pytest

from test_gpu_binning import _screen
from test_gpu_binning_sizes import _binned

pytestmark = pytest.mark.gpu

CHUNKS = 1824    # most chunks of a size below 2,048


@pytest.mark.parametrize("size,n,W,H,rmax", [(256, 200_000, 1600, 900, 40), (512, 300_000, 1600, 900, 40),
                                             (1024, 500_000, 1920, 1080, 60), (2048, 800_000, 1920, 1080, 60)])
def test_each_chunk_size(size, n, W, H, rmax):
    sp = _screen(170, n, W, H, rmax, huge=2)
    a, b = (_binned(sp, W, H, mode, 24_000_000) for mode in ("two_phase", "key64"))
    records = a[1]
    assert records <= size * CHUNKS or size == 2048
    assert records > size // 2 * CHUNKS or size == 256
    assert a[0] == b[0] and a[1] == b[1]
    for x, y in zip(a[2:], b[2:]):
        assert np.array_equal(x, y)
