"""The one-block depth sort skips a byte pass when the byte is the same in every key: all Gaussians
at one depth, depths that agree in one or two bytes, all of them culled, or a single one.  Skipped
and taken passes follow one another in every combination, over a partial warp, one, several and all
items per thread; every repetition gives the same lists, each in the order of a stable sort by depth
and index, and equal to those of the KEY64 schedule, whose passes skip nothing."""
import numpy as np
import pytest

from test_gpu_binning import _frame, _screen

pytestmark = pytest.mark.gpu

W, H, CAPACITY, REPEATS = 333, 251, 1 << 18, 200


def _depths(free, n, seed):
    """Positive finite depths whose bits vary in the bytes `free` only (0: the lowest)."""
    rng = np.random.default_rng(seed)
    bits = np.full(n, 0x40200000, np.uint32)     # 2.5
    for byte in free:
        vary = rng.integers(0x3E, 0x42, n) if byte == 3 else rng.integers(0, 256, n)
        bits &= np.uint32(~(0xFF << 8 * byte) & 0xFFFFFFFF)
        bits |= vary.astype(np.uint32) << np.uint32(8 * byte)
    return bits.view(np.float32)


FREE = [(), (0,), (1,), (2,), (3,), (0, 1), (0, 2), (1, 2), (0, 3), (0, 1, 3), (0, 2, 3), (1, 2, 3)]


def _check(sp):
    import torch
    n = len(sp["depth"])
    want = _frame(sp, W, H, (16, 16), "key64", CAPACITY)
    want.bin_sort()
    code, st = want.status()
    assert code == 0
    K = int(st.num_instances)
    wvals = want.view("vals_sorted", torch.int32, max(K, 1))[:K]
    wranges = want.view("ranges", torch.int32, 2 * want.tiles)
    vals, ranges = wvals.cpu().numpy().astype(np.int64), wranges.cpu().numpy().reshape(-1, 2)
    key = np.where(sp["radius"] > 0, sp["depth"].view(np.uint32), np.uint32(0xFFFFFFFF))
    rank = np.empty(n, np.int64)
    rank[np.argsort(key, kind="stable")] = np.arange(n)
    for a, b in ranges:
        assert np.all(np.diff(rank[vals[a:b]]) > 0)
    fr = _frame(sp, W, H, (16, 16), "two_phase", CAPACITY)
    for _ in range(REPEATS):
        fr.view("vals_sorted", torch.int32, max(K, 1)).fill_(-1)
        fr.bin_sort()
        assert torch.equal(fr.view("ranges", torch.int32, 2 * fr.tiles), wranges)
        assert torch.equal(fr.view("vals_sorted", torch.int32, max(K, 1))[:K], wvals)
    code, st = fr.status()
    assert code == 0 and int(st.num_instances) == K
    return K


@pytest.mark.parametrize("free", FREE, ids=str)
@pytest.mark.parametrize("n", [33, 1000, 5000, 8192])
def test_bytes_that_every_key_shares(n, free):
    sp = _screen(300 + n, n, W, H, 12, culled=0.0, ties=0.0)
    sp["depth"] = _depths(free, n, n)
    for byte in range(4):
        assert (np.unique(sp["depth"].view(np.uint32) >> np.uint32(8 * byte) & 0xFF).size == 1) == (byte not in free)
    assert _check(sp) > 0


@pytest.mark.parametrize("n", [1, 33, 5000, 8192])
def test_all_culled(n):
    sp = _screen(320 + n, n, W, H, 12, culled=1.0)
    assert _check(sp) == 0


def test_a_single_gaussian():
    sp = _screen(331, 1, W, H, 12, culled=0.0)
    sp["uv"][:] = 100.0
    assert _check(sp) > 0
