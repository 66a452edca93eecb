"""The graph loop unrolls several iterations per round of its while-node and
the host loop's launches run ahead of the condition it reads back: a run ends
at its budget, skipped launches change nothing, and a single step after a
finished run still steps. Histories against the oracle: integer counts exact,
deposits to 1e-9."""
import numpy as np
import pytest

from paper_2503_17608_gb300 import binding, workloads as wl

from gpu_helpers import match_fraction, run_oracle

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("policy", [wl.SORT_NONE, wl.SORT_ACTION_TYPE, wl.SORT_LOCAL, wl.SORT_DATA])
@pytest.mark.parametrize("budget", [1, 3, 4, 5, 8, 0])
def test_graph_runs_end_at_their_budget(policy, budget):
    prim = wl.electron_beam(40, 200.0)
    prob = wl.calorimeter_problem(2048, history_capacity=40, sort_policy=policy)
    with binding.Context(prob) as ctx:
        ctx.add_primaries(0, prim)
        total, runs = 0, 0
        while True:
            done = ctx.run_iterations(binding.LOOP_GRAPH, budget=budget)
            total += done
            runs += 1
            s = ctx.stats()
            assert s["iteration"] == total
            if s["alive"] == 0 and s["queued"] == 0:
                break
            assert budget and done == budget
        assert budget == 0 or done <= budget
        hist, edep = ctx.read_history(0, len(prim))
    assert runs == (1 if budget == 0 else -(-total // budget))
    frac, _ = match_fraction(dict(hist=hist, edep=edep), run_oracle(prob, prim))
    assert frac == 1.0, frac


@pytest.mark.parametrize("policy", [wl.SORT_NONE, wl.SORT_ACTION, wl.SORT_LOCAL])
@pytest.mark.parametrize("hits", [0, 1])
def test_steps_after_a_finished_run(policy, hits):
    """Runs to the end in the host and the graph loop, single steps in between
    that find new primaries, and a run with nothing to do."""
    import torch

    n = 64
    prob = wl.water_cube_problem(n_slots=512, history_capacity=4 * n, sort_policy=policy)
    prim = wl.water_cube_primaries(n)
    with binding.Context(prob) as ctx:
        if hits:
            buf = torch.zeros(prob.max_events * ctx.n_bins, dtype=torch.float64).pin_memory()
            ctx.set_hit_readout(1, buf)
        for k, mode in enumerate([binding.LOOP_HOST, binding.LOOP_GRAPH, binding.LOOP_HOST, binding.LOOP_GRAPH]):
            prim["event"][:] = k
            ctx.add_primaries(k, prim)
            before = ctx.stats()["steps_total"]
            ctx.step()
            assert ctx.stats()["steps_total"] == before + n  # every primary took its first step
            ctx.run_events(mode)
            s = ctx.stats()
            assert s["alive"] == 0 and s["queued"] == 0
            ctx.run_events(mode)  # nothing to do
            assert ctx.stats()["steps_total"] == s["steps_total"] and ctx.stats()["iteration"] == s["iteration"]
            if hits and mode == binding.LOOP_HOST:
                tally = np.concatenate([ctx.read_tallies(e)[0] for e in range(prob.max_events)])
                np.testing.assert_array_equal(buf.numpy(), tally)
        hist, edep = ctx.read_history(0, 4 * n)
    for k in range(4):
        prim["event"][:] = k
        frac, _ = match_fraction(dict(hist=hist[k * n:(k + 1) * n], edep=edep[k * n:(k + 1) * n]), run_oracle(prob, prim))
        assert frac == 1.0, (k, frac)
