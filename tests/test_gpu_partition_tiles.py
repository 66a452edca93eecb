"""The allocation-free key partition at the edges of its tiles (4,096 slots, 16
keys per thread), with unaligned key arrays, keys out of range and a skipped
key, against numpy's stable argsort. Whole numbers: exact."""
import numpy as np
import pytest

from paper_2503_17608_gb300 import binding

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [1, 15, 16, 17, 4095, 4096, 4097, 8192, 8193, 65536 + 5, (1 << 20) - 1, 1 << 20])
@pytest.mark.parametrize("n_keys,skip,offset", [(1, -1, 0), (9, 8, 0), (16, 3, 1), (7, -1, 3)])
def test_partition_at_tile_edges(n, n_keys, skip, offset):
    import torch

    rng = np.random.default_rng(n * 31 + n_keys)
    keys = rng.integers(0, n_keys + 2, n).astype(np.uint8)  # some out of range
    keys[rng.uniform(size=n) < 0.5] = n_keys - 1
    buf = torch.zeros(n + 16, dtype=torch.uint8, device="cuda")
    buf[offset : offset + n] = torch.from_numpy(keys).cuda()
    perm = torch.full((n,), -1, dtype=torch.int32, device="cuda")
    offs = torch.full((n_keys + 1,), -1, dtype=torch.int32, device="cuda")
    binding.partition_keys_noalloc(buf.data_ptr() + offset, n, n_keys, skip, perm.data_ptr(), offs.data_ptr(),
                                   torch.cuda.current_stream().cuda_stream)
    counts = np.bincount(keys, minlength=n_keys + 2)[:n_keys]
    want_offs = np.concatenate([[0], np.cumsum(counts)])
    want = np.full(n, -1)
    order = np.argsort(keys, kind="stable")[: want_offs[-1]]
    want[: len(order)] = order
    if skip >= 0:
        want[want_offs[skip] : want_offs[skip + 1]] = -1
    np.testing.assert_array_equal(offs.cpu().numpy(), want_offs)
    np.testing.assert_array_equal(perm.cpu().numpy(), want)
