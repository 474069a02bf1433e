"""The two-phase schedule changes its layout with the frame's size: a frame of at most 8,192
Gaussians is depth-sorted by one block, the radix passes take 4, 8 or 16 keys per thread by the number
of keys, and the column passes 256 to 2,048 records per chunk by the number of records of the launch.  At the edges of these ranges the result is that of the
KEY64 schedule, which shares none of it, bit for bit."""
import numpy as np
import pytest

import synthetic as S
from test_gpu_binning import _frame, _screen

pytestmark = pytest.mark.gpu


def _binned(sp, W, H, mode, capacity):
    import torch
    fr = _frame(sp, W, H, (16, 16), mode, capacity)
    fr.bin_sort()
    code, st = fr.status()
    assert code == 0
    K = int(st.num_instances)
    ranges = fr.view("ranges", torch.int32, 2 * fr.tiles).cpu().numpy()
    vals = fr.view("vals_sorted", torch.int32, max(K, 1)).cpu().numpy()[:K]
    order = fr.view("tile_order", torch.int32, fr.tiles).cpu().numpy()
    return K, int(st.num_segments), ranges, vals, order


@pytest.mark.parametrize("n", [1, 2, 31, 33, 1023, 1024, 1025, 2049, 8191, 8192, 8193])
def test_depth_order_of_small_frames(n):
    sp = _screen(100 + n, n, 333, 251, 12, culled=0.2, ties=0.3)
    a, b = (_binned(sp, 333, 251, mode, 1 << 18) for mode in ("two_phase", "key64"))
    assert a[0] == b[0]
    for x, y in zip(a[2:], b[2:]):
        assert np.array_equal(x, y)


def test_depth_order_where_a_byte_is_shared_or_all_depths_are_equal():
    for depth in (np.full(3000, 2.5, np.float32), np.float32(2.0) + np.arange(3000, dtype=np.float32)[::-1] * 1e-6):
        sp = _screen(140, 3000, 333, 251, 12, culled=0.1)
        sp["depth"] = np.ascontiguousarray(depth)
        a, b = (_binned(sp, 333, 251, mode, 1 << 18) for mode in ("two_phase", "key64"))
        assert a[0] == b[0] and all(np.array_equal(x, y) for x, y in zip(a[2:], b[2:]))


# records of the launch below and above each change of the chunk size (256 x 1824 x 1, 2, 4)
@pytest.mark.parametrize("n,W,H,rmax", [(9000, 640, 480, 6), (90_000, 1280, 720, 40), (200_000, 1600, 900, 40),
                                        (330_000, 1920, 1080, 60), (500_000, 1920, 1080, 60)])
def test_column_chunk_sizes(n, W, H, rmax):
    sp = _screen(150, n, W, H, rmax, huge=2)
    cap = 24_000_000
    a, b = (_binned(sp, W, H, mode, cap) for mode in ("two_phase", "key64"))
    assert a[0] == b[0] and a[1] == b[1]
    for x, y in zip(a[2:], b[2:]):
        assert np.array_equal(x, y)
    print(f"n {n}: {a[1]} records, {a[0]} instances")


@pytest.mark.parametrize("n", [1 << 18, (1 << 18) + 1, (1 << 20) - 3, (1 << 20) + 1])
def test_depth_passes_where_the_keys_per_thread_change(n):
    sp = _screen(160, n, 640, 480, 4, culled=0.3, ties=0.3)
    a, b = (_binned(sp, 640, 480, mode, 6_000_000) for mode in ("two_phase", "key64"))
    assert a[0] == b[0] and a[1] == b[1]
    for x, y in zip(a[2:], b[2:]):
        assert np.array_equal(x, y)


@pytest.mark.parametrize("capacity", [6_000_000, 6_000_001])
def test_two_row_passes_in_either_kernel(capacity):
    # over 256 tile rows: two row passes, with the keys per thread chosen on the device or fixed
    sp = _screen(161, 60_000, 300, 4400, 60)
    a, b = (_binned(sp, 300, 4400, mode, capacity) for mode in ("two_phase", "key64"))
    assert a[0] == b[0] and a[1] == b[1]
    for x, y in zip(a[2:], b[2:]):
        assert np.array_equal(x, y)
