"""The per-warp schedule's shared-memory track store: its small variant (many
materials leave room for fewer tracks per block), tracks left between two
steps by budgeted runs and taken up again by every loop, and events whose ids
exceed the tally rows. Every history against the oracle, as in the other
asynchronous tests: integer counts exact, deposits to 1e-9."""
import numpy as np
import pytest

from paper_2503_17608_gb300 import binding, workloads as wl

from gpu_helpers import assert_conservation, match_fraction, run_gpu, run_oracle

pytestmark = pytest.mark.gpu


def oracle_check(prob, prim, hist, edep):
    frac, _ = match_fraction(dict(hist=hist, edep=edep), run_oracle(prob, prim))
    assert frac == 1.0, frac


@pytest.mark.parametrize("n_materials", [4, 5, 8])
def test_many_materials(n_materials):
    """Four materials fit beside 1,024 tracks, eight beside 256; tracks cross
    all of them, so the flight's two kept cross sections are replaced often."""
    base = wl.calorimeter_problem(8192)
    mats = [wl.LEAD if i % 2 == 0 else wl.LAR for i in range(n_materials)]
    prob = base.replace(materials=mats, layer_material=list(range(n_materials)),
                        layer_thickness=[0.2 if i % 2 == 0 else 0.5 for i in range(n_materials)],
                        n_periods=80 // n_materials, sort_policy=wl.SORT_LOCAL)
    prim = wl.electron_beam(200, 1000.0)
    g = run_gpu(prob, prim, mode=binding.LOOP_ASYNC)
    oracle_check(prob, prim, g["hist"], g["edep"])


@pytest.mark.parametrize("bz,cap", [(0.0, 0), (4.0, 0), (4.0, 10)])
@pytest.mark.parametrize("half", [2.0, 50.0])
def test_budgeted_runs_of_showers_interleaved_with_other_loops(bz, cap, half):
    """Electrons and photons stored between two steps (grid positions, pending
    interactions and all), taken up by other loops and back."""
    rng = np.random.default_rng(3)
    prim = wl.electron_beam(120, 500.0, patch_half=min(half, 5.0) * 0.9)
    prim["ptype"][::3] = wl.GAMMA
    d = rng.normal(size=(120, 3))
    d[:, 2] = np.abs(d[:, 2]) + 0.3
    prim["dir"] = d / np.linalg.norm(d, axis=1, keepdims=True)
    prob = wl.calorimeter_problem(4096, Bz=bz, half_x=half, half_y=half, field_substep_cap=cap, history_capacity=120,
                                  sort_policy=wl.SORT_LOCAL)
    others = [(wl.SORT_LOCAL, binding.LOOP_PERSISTENT), (wl.SORT_DATA, binding.LOOP_ASYNC),
              (wl.SORT_ACTION_TYPE, binding.LOOP_GRAPH), (wl.SORT_NONE, binding.LOOP_HOST)]
    with binding.Context(prob) as ctx:
        ctx.add_primaries(0, prim)
        for k in range(400):
            ctx.set_sort_policy(wl.SORT_LOCAL)
            ctx.run_iterations(binding.LOOP_ASYNC, budget=2)
            policy, mode = others[k % len(others)]
            ctx.set_sort_policy(policy)
            ctx.run_iterations(mode, budget=2)
            s = ctx.stats()
            if s["alive"] == 0 and s["queued"] == 0:
                break
        hist, edep = ctx.read_history(0, len(prim))
    assert s["alive"] == 0 and s["queued"] == 0 and k > 2
    oracle_check(prob, prim, hist, edep)


def test_event_ids_beyond_the_tally_rows():
    prob = wl.calorimeter_problem(4096, max_events=3, sort_policy=wl.SORT_LOCAL)
    prim = wl.electron_beam(60, 300.0, event=1000)
    prim["event"][30:] = 7001
    g = run_gpu(prob, prim, mode=binding.LOOP_ASYNC)
    o = run_oracle(prob, prim)
    oracle_check(prob, prim, g["hist"], g["edep"])
    for e in (1000, 7001):
        want = o["edep"][prim["event"] == e].sum(0)
        np.testing.assert_allclose(g["tally"][e][0], want, rtol=0, atol=1e-9 * want.max())


@pytest.mark.parametrize("n", [1, 255, 257, 4097])
def test_queued_primaries_between_runs_of_all_loops(n):
    """Runs of the asynchronous loop take up the buffer as the last run and the
    pushes since left it; synchronous runs in between make them set it up
    anew. Host batches below and above the size read in place, device batches,
    and a budgeted run in the middle."""
    import torch

    # (room for two batches: a budgeted run leaves most of its own queued)
    prob = wl.water_cube_problem(n_slots=2048, init_capacity=16384, history_capacity=8 * n, sort_policy=wl.SORT_LOCAL)
    runs = [(wl.SORT_LOCAL, binding.LOOP_ASYNC, 0), (wl.SORT_LOCAL, binding.LOOP_ASYNC, 2),
            (wl.SORT_DATA, binding.LOOP_ASYNC, 0), (wl.SORT_LOCAL, binding.LOOP_ASYNC, 0),
            (wl.SORT_NONE, binding.LOOP_PERSISTENT, 3), (wl.SORT_LOCAL, binding.LOOP_ASYNC, 0)]
    prim = wl.water_cube_primaries(n)
    dev = torch.from_numpy(binding.to_c_primaries(prim).view(np.uint8).copy()).cuda()
    with binding.Context(prob) as ctx:
        for k, (policy, mode, budget) in enumerate(runs):
            ctx.set_sort_policy(policy)
            if k % 2:
                ctx.add_primaries_device(k, dev.data_ptr(), n)
            else:
                prim["event"][:] = k
                ctx.add_primaries(k, prim)
            ctx.run_iterations(mode, budget=budget)
        s = ctx.stats()
        assert s["alive"] == 0 and s["queued"] == 0
        hist, edep = ctx.read_history(0, len(runs) * n)
    for k in range(len(runs)):
        prim["event"][:] = k
        o = run_oracle(prob, prim)
        np.testing.assert_array_equal(hist["steps"][k * n:(k + 1) * n], o["hist"]["steps"])
        np.testing.assert_allclose(edep[k * n:(k + 1) * n], o["edep"], rtol=1e-9, atol=1e-9 * 10.0)


@pytest.mark.parametrize("n,energy", [(96000, 5.0), (120000, 20.0), (160000, 1.0)])
def test_blocks_that_hold_many_tracks(n, energy):
    """640 tracks a block and more (97,280 on 152 blocks): only full pieces are
    taken until the number falls below it, small ones after that."""
    prob = wl.calorimeter_problem(1 << 18, Bz=4.0, init_capacity=1 << 18, history_capacity=n, sort_policy=wl.SORT_LOCAL)
    prim = wl.electron_beam(n, energy, patch_half=5.0)
    prim["ptype"][1::2] = wl.GAMMA
    g = run_gpu(prob, prim, mode=binding.LOOP_ASYNC)
    oracle_check(prob, prim, g["hist"], g["edep"])


@pytest.mark.parametrize("policy", [wl.SORT_LOCAL, wl.SORT_DATA])
@pytest.mark.parametrize("capacity", [4096, 8192, 16384])
def test_buffer_smaller_than_the_shower(policy, capacity):
    """The buffer's free entries run out: groups of lanes get none or some of
    what they ask for, and the interactions without one wait for room."""
    prob = wl.calorimeter_problem(1 << 15, Bz=4.0, init_capacity=capacity, sort_policy=policy)
    prim = wl.electron_beam(3000, 200.0, patch_half=5.0)
    g = run_gpu(prob, prim, mode=binding.LOOP_ASYNC)
    oracle_check(prob, prim, g["hist"], g["edep"])
    assert_conservation(prim, g["tally"], rel=1e-11)
