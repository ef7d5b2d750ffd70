"""The event schedule with more bins than its shared-memory tables hold by
default (3072 and more asked for over 48 KiB, which no launch was given)."""
import numpy as np
import pytest

from paper_2403_06362_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("bins", [3070, 3071, 3072, 4095, 4096])
def test_event_schedule_matches_the_history_schedule(bins):
    import paper_2403_06362_gb300 as mc
    ctx = mc.Context(0)
    p = [W.slab_problem(10.0, 1.0, 0.8, 1000, bins, 1, W.SEED_HASH)]
    out = []
    for schedule in (mc.MC_SCHED_HISTORY, mc.MC_SCHED_EVENT):
        t = mc.Tally(W.tally_slots(p), 1)
        mc.mc_transport_run(ctx, mc.make_lcg(), [W.to_mc_problem(q, mc) for q in p],
                            mc.mc_run_config(schedule=schedule), t.c)
        out.append((t.bins.cpu().numpy(), t.counts.cpu().numpy()))
    assert np.array_equal(out[0][0], out[1][0]) and np.array_equal(out[0][1], out[1][1])
    ctx.close()
