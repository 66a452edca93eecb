"""A context that cannot be created (its buffer is larger than the device)
leaves nothing behind that the calls of other contexts would report."""
import pytest

from paper_2503_17608_gb300 import binding, workloads as wl

pytestmark = pytest.mark.gpu


def test_other_contexts_work_after_a_failed_creation():
    prim = wl.water_cube_primaries(50)
    with binding.Context(wl.water_cube_problem(n_slots=1024, sort_policy=wl.SORT_LOCAL)) as ctx:
        ctx.add_events(prim)
        ctx.run_events(binding.LOOP_ASYNC)

        def fail():
            with pytest.raises(binding.CelerError) as ei:
                binding.Context(wl.water_cube_problem(n_slots=1024, init_capacity=1 << 34))
            assert ei.value.status == 3  # CELER_ERR_CUDA: 1.4 TB asked of one device

        # each call first thing after a failure
        fail()
        tally, esc = ctx.read_tallies(0)
        assert tally.sum() + esc == pytest.approx(prim["E"].sum(), rel=1e-12)
        fail()
        assert ctx.stats()["alive"] == 0
        fail()
        ctx.reset_event(0)
        fail()
        ctx.add_events(prim)
        fail()
        ctx.run_events(binding.LOOP_ASYNC)
        fail()
        tally, esc = ctx.read_tallies(0)
        assert tally.sum() + esc == pytest.approx(prim["E"].sum(), rel=1e-12)
