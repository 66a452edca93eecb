"""Tracks that a budgeted per-warp run takes from the buffer and still holds at
its end go into its block's vacant slots, shared out among the block's warps:
each track into one slot, and the counts of the slots with them."""
import numpy as np
import pytest

from paper_2503_17608_gb300 import binding, workloads as wl

from gpu_helpers import match_fraction, run_oracle

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("blocks,n_slots", [(1, 1024), (2, 1216), (2, 2000), (3, 5001)])
def test_every_track_in_one_slot_after_each_chunk(blocks, n_slots):
    """Few blocks, so that all sixteen warps of each store at once, into slots
    of which most are taken, with a part-filled last chunk."""
    n = 4000
    prob = wl.water_cube_problem(n_slots=n_slots, history_capacity=n, sort_policy=wl.SORT_LOCAL)
    prim = wl.water_cube_primaries(n)
    held = 0
    with binding.Context(prob) as ctx:
        ctx.set_grid_blocks(blocks)
        ctx.add_events(prim)
        for run in range(2000):
            ctx.run_iterations(binding.LOOP_ASYNC, budget=4)
            s = ctx.stats()
            live = ctx.debug_slots()["status"] != 0
            assert live.sum() == s["alive"]
            tids = ctx.debug_tracks()["tid"][live]
            assert len(np.unique(tids)) == len(tids)
            held = max(held, int(live.sum()))
            if s["alive"] == 0 and s["queued"] == 0:
                break
        hist, edep = ctx.read_history(0, n)
    assert s["alive"] == 0 and s["queued"] == 0 and run > 3
    assert held > 32
    frac, _ = match_fraction(dict(hist=hist, edep=edep), run_oracle(prob, prim))
    assert frac == 1.0, frac
