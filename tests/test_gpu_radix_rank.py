"""The radix passes find a warp's lanes of one digit in three ways: one word per digit in shared
memory, no words where the whole warp holds one digit, and match_any for the top byte.  The order
is the host's stable sort of the keys, index for index, for keys that are spread, equal, few, or
mostly culled, with partial warps and chunks at the end."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

KINDS = {
    "spread": lambda rng, n: rng.uniform(0.2, 30.0, n),
    "equal": lambda rng, n: np.full(n, 2.5),
    "few": lambda rng, n: rng.choice([0.25, 0.5, 3.0, 3.0000002, 700.0], n),
    "runs": lambda rng, n: np.repeat(rng.uniform(1.0, 4.0, n // 40 + 1), 40)[:n],
    "all bits": lambda rng, n: rng.integers(1, 0x7F7FFFFF, n).astype(np.uint32).view(np.float32),
}


@pytest.mark.parametrize("kind", sorted(KINDS))
@pytest.mark.parametrize("n,culled", [(1, 0.0), (33, 0.5), (4097, 0.2), (100_003, 0.9), (262_144, 0.1)])
def test_depth_order_is_the_stable_sort(kind, n, culled):
    import torch
    from paper_2308_04079_gb300 import _abi
    rng = np.random.default_rng(n)
    depth = np.ascontiguousarray(KINDS[kind](rng, n), dtype=np.float32)
    radius = np.where(rng.random(n) < culled, -rng.integers(0, 2, n), rng.integers(1, 9, n)).astype(np.int32)
    d, r = torch.from_numpy(depth).cuda(), torch.from_numpy(radius).cuda()
    order = torch.full((n,), -1, dtype=torch.int32, device="cuda")
    status = torch.full((8,), -1, dtype=torch.int32, device="cuda")
    _abi.gs_depth_order_static(n, d.data_ptr(), r.data_ptr(), order.data_ptr(), status.data_ptr(),
                               torch.cuda.current_stream().cuda_stream)
    torch.cuda.synchronize()
    key = np.where(radius > 0, depth.view(np.uint32), np.uint32(0xFFFFFFFF))
    assert np.array_equal(order.cpu().numpy(), np.argsort(key, kind="stable"))
    st = status.cpu().numpy().view(np.uint32)
    assert st[0] == 0 and st[2] == np.count_nonzero(radius > 0)
