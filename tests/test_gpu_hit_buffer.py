"""Per-iteration hit readout into any pinned buffer: whole pages, parts of
them, and one that does not start on a double's boundary (copied instead of
written by the kernels)."""
import numpy as np
import pytest

from paper_2503_17608_gb300 import binding, workloads as wl

pytestmark = pytest.mark.gpu


class Bytes:
    """n doubles at a byte offset of a pinned tensor of bytes."""

    def __init__(self, raw, offset, n):
        self.raw, self.offset, self.n = raw, offset, n

    def data_ptr(self):
        return self.raw.data_ptr() + self.offset

    def numel(self):
        return self.n

    def values(self):
        return np.frombuffer(self.raw.numpy().tobytes(), np.float64, self.n, self.offset)


@pytest.mark.parametrize("offset", [0, 8, 4088, 4, 4093])
@pytest.mark.parametrize("max_events,n_zbins", [(1, 1), (3, 50), (8, 512), (9, 512)])
def test_hits_at_any_offset(offset, max_events, n_zbins):
    import torch

    prob = wl.water_cube_problem(n_slots=1024, max_events=max_events).replace(n_zbins=n_zbins)
    prim = wl.water_cube_primaries(100)
    with binding.Context(prob) as ctx:
        n = max_events * ctx.n_bins
        raw = torch.zeros(8 * n + 8192, dtype=torch.uint8).pin_memory()
        hits = Bytes(raw, offset, n)
        ctx.set_hit_readout(1, hits)
        ctx.add_events(prim)
        ctx.run_events(binding.LOOP_HOST)
        want = np.concatenate([ctx.read_tallies(e)[0] for e in range(max_events)])
        np.testing.assert_array_equal(hits.values(), want)
    assert want.sum() > 0
    assert not raw[:offset].any() and not raw[offset + 8 * n:].any()
