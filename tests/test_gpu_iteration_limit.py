"""Asynchronous runs that end at the iteration limit (passes of a block, pieces
of a warp) while other blocks are in the middle of theirs: the run reports the
status, every claimed buffer entry is read and every reserved one written, and
the next runs go on from the state it left, so that after enough of them every
history is the oracle's."""
import numpy as np
import pytest

from paper_2503_17608_gb300 import binding, workloads as wl

from gpu_helpers import assert_conservation, match_fraction, run_oracle

pytestmark = pytest.mark.gpu

SCHEDULES = [(wl.SORT_LOCAL, True), (wl.SORT_LOCAL, False), (wl.SORT_DATA, False)]
SCHED_IDS = ["local-warps", "local-passes", "data-passes"]


@pytest.mark.parametrize("policy,warps", SCHEDULES, ids=SCHED_IDS)
@pytest.mark.parametrize("limit,capacity", [(1, 1 << 16), (5, 1 << 16), (40, 4096)])
def test_runs_cut_off_by_the_limit_lose_nothing(policy, warps, limit, capacity):
    n = 300
    prob, prim = wl.calorimeter_1gev(n)
    prob = prob.replace(n_slots=1 << 15, init_capacity=capacity, history_capacity=n, sort_policy=policy)
    with binding.Context(prob, max_iterations=limit) as ctx:
        ctx.set_async_warps(warps)
        ctx.add_events(prim)
        for run in range(20000):
            with pytest.raises(binding.CelerError) as ei:
                ctx.run_events(binding.LOOP_ASYNC)
            assert ei.value.status == 4  # CELER_ERR_TIMEOUT
            s = ctx.stats()
            live = ctx.debug_slots()["status"] != 0
            assert live.sum() == s["alive"]
            if s["alive"] == 0 and s["queued"] == 0:
                break
        assert s["alive"] == 0 and s["queued"] == 0
        assert s["error"] == 4  # the iteration limit's bit alone: no wait gave up
        hist, edep = ctx.read_history(0, n)
        tally = {0: ctx.read_tallies(0)}
    frac, _ = match_fraction(dict(hist=hist, edep=edep), run_oracle(prob, prim))
    assert frac == 1.0, frac
    assert_conservation(prim, tally, rel=1e-11)
