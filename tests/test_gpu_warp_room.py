"""Blocks of the per-warp schedule that hold more tracks than their shared
memory has entries: with the buffer full and every entry's track waiting for
room in it, tracks move to vacant slots until there is room again. Histories
equal those of the synchronous loop with a buffer that never fills."""
import numpy as np
import pytest

from paper_2503_17608_gb300 import binding, workloads as wl

from gpu_helpers import assert_conservation, run_gpu

pytestmark = pytest.mark.gpu


def world(n_materials, **kw):
    mats = [wl.LEAD if i % 2 == 0 else wl.LAR for i in range(n_materials)]
    return wl.calorimeter_problem(1 << 15, sort_policy=wl.SORT_LOCAL, **kw).replace(
        materials=mats, layer_material=list(range(n_materials)),
        layer_thickness=[0.2 if i % 2 == 0 else 0.5 for i in range(n_materials)], n_periods=80 // n_materials)


def check(prob, prim, hist, edep, tally):
    s = run_gpu(prob.replace(init_capacity=1 << 19), prim, mode=binding.LOOP_PERSISTENT)
    np.testing.assert_array_equal(hist["steps"], s["hist"]["steps"])
    np.testing.assert_array_equal(hist["secondaries"], s["hist"]["secondaries"])
    np.testing.assert_allclose(edep, s["edep"], rtol=1e-12, atol=1e-12)
    assert_conservation(prim, tally, rel=1e-11)


# entries of eight blocks: 8,192 with two materials, less with more
@pytest.mark.parametrize("n_materials,n,capacity", [(2, 9000, 1 << 14), (5, 9000, 1 << 14), (6, 3000, 4096),
                                                    (8, 3000, 4096), (8, 9000, 1 << 14)])
@pytest.mark.parametrize("budget", [0, 50])
def test_full_buffer_and_all_entries_waiting(n_materials, n, capacity, budget):
    prob = world(n_materials, init_capacity=capacity, history_capacity=n)
    prim = wl.electron_beam(n, 150.0, patch_half=5.0)
    with binding.Context(prob) as ctx:
        ctx.set_grid_blocks(8)
        ctx.add_events(prim)
        for _ in range(5000):
            ctx.run_iterations(binding.LOOP_ASYNC, budget=budget)
            s = ctx.stats()
            assert (ctx.debug_slots()["status"] != 0).sum() == s["alive"]
            if s["alive"] == 0 and s["queued"] == 0:
                break
        assert s["alive"] == 0 and s["queued"] == 0
        hist, edep = ctx.read_history(0, n)
        tally = {0: ctx.read_tallies(0)}
    check(prob, prim, hist, edep, tally)


# (the last two: no slot to spare; the entries' tracks make way for parked ones that can move)
@pytest.mark.parametrize("n_materials,blocks,n_slots,energy,before",
                         [(2, 2, 1 << 15, 150.0, 8), (2, 2, 1 << 15, 150.0, 25), (8, 8, 1 << 15, 150.0, 8),
                          (8, 8, 1 << 15, 150.0, 25), (2, 2, 4096, 20.0, 10), (8, 4, 4096, 20.0, 25)])
def test_more_live_tracks_than_entries_at_the_start_and_a_full_buffer(n_materials, blocks, n_slots, energy, before):
    n = 4000
    prob = world(n_materials, init_capacity=4096, history_capacity=n).replace(n_slots=n_slots)
    prim = wl.electron_beam(n, energy, patch_half=5.0)
    with binding.Context(prob) as ctx:
        ctx.set_grid_blocks(blocks)
        ctx.add_events(prim)
        ctx.run_iterations(binding.LOOP_PERSISTENT, budget=before)
        assert ctx.stats()["alive"] > 2048
        ctx.run_events(binding.LOOP_ASYNC)
        s = ctx.stats()
        assert s["alive"] == 0 and s["queued"] == 0
        hist, edep = ctx.read_history(0, n)
        tally = {0: ctx.read_tallies(0)}
    check(prob.replace(n_slots=1 << 15), prim, hist, edep, tally)


@pytest.mark.parametrize("n_materials,n_periods", [(5, 52), (5, 53), (6, 13), (8, 82), (8, 83), (8, 128)])
def test_as_many_entries_as_fit_beside_the_tables(n_materials, n_periods):
    """Worlds on both sides of the lines between 1,024, 512 and 256 entries
    (261 layers of five materials, 658 of eight), four blocks with more tracks
    than the number from which on they take full pieces only."""
    n = 3000
    prob = world(n_materials, init_capacity=1 << 18, history_capacity=n).replace(
        n_periods=n_periods, layer_thickness=[0.1 if i % 2 == 0 else 0.25 for i in range(n_materials)])
    prim = wl.electron_beam(n, 100.0, patch_half=5.0)
    with binding.Context(prob) as ctx:
        ctx.set_grid_blocks(4)
        ctx.add_events(prim)
        ctx.run_events(binding.LOOP_ASYNC)
        s = ctx.stats()
        assert s["alive"] == 0 and s["queued"] == 0
        hist, edep = ctx.read_history(0, n)
        tally = {0: ctx.read_tallies(0)}
    check(prob, prim, hist, edep, tally)
