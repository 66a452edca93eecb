"""Block passes of the asynchronous loop with a buffer that their own claims
reach around: a block reads all the entries it has claimed before its first
step, so none of its writers waits for one of them. Histories equal those of
the synchronous loop with a buffer that never fills."""
import numpy as np
import pytest

from paper_2503_17608_gb300 import binding, workloads as wl

from gpu_helpers import assert_conservation, run_gpu

pytestmark = pytest.mark.gpu


# (two blocks of 4,096 and 2,048 slots: one batch of chunks each; of 16,384: two)
@pytest.mark.parametrize("policy", [wl.SORT_LOCAL, wl.SORT_DATA])
@pytest.mark.parametrize("n_slots,before", [(8192, 4), (8192, 10), (4096, 4), (4096, 25), (1 << 15, 4), (4096 + 33, 10)])
def test_claims_that_reach_around_the_buffer(policy, n_slots, before):
    n = 4000
    prob = wl.calorimeter_problem(n_slots, Bz=4.0, init_capacity=4096, history_capacity=n, sort_policy=policy)
    prim = wl.electron_beam(n, 20.0, patch_half=5.0)
    with binding.Context(prob) as ctx:
        ctx.set_grid_blocks(2)
        ctx.set_async_warps(False)
        ctx.add_events(prim)
        ctx.run_iterations(binding.LOOP_PERSISTENT, budget=before)
        ctx.run_events(binding.LOOP_ASYNC)
        s = ctx.stats()
        assert s["alive"] == 0 and s["queued"] == 0 and s["error"] == 0
        hist, edep = ctx.read_history(0, n)
        tally = {0: ctx.read_tallies(0)}
    s = run_gpu(prob.replace(init_capacity=1 << 17, n_slots=1 << 15), prim, mode=binding.LOOP_PERSISTENT)
    np.testing.assert_array_equal(hist["steps"], s["hist"]["steps"])
    np.testing.assert_array_equal(hist["secondaries"], s["hist"]["secondaries"])
    np.testing.assert_allclose(edep, s["edep"], rtol=1e-12, atol=1e-12)
    assert_conservation(prim, tally, rel=1e-11)
