"""Long histories over more bins than any block stages, fewer of them than a
warp has lanes and a few more, where the last lanes of a warp walk their bins
together: the bits of the event schedule, which keeps no walk between passes."""
import pytest

from paper_2403_06362_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("seeding", [W.SEED_HASH, W.SEED_STRIDE])
@pytest.mark.parametrize("n", [1, 7, 8, 9, 40])
def test_schedules_agree(n, seeding, precision):
    import torch

    import paper_2403_06362_gb300 as mc

    ctx = mc.Context(0)
    p = W.slab_problem(60.0, 1.0, 0.999, n, 9000, 1, seeding)
    out = []
    for cfg in (dict(), dict(block=32, chunk=4), dict(block=256, tally_atomics=2), dict(schedule=1)):
        t = mc.Tally(W.tally_slots([p]), 1, n_histories=n)
        mc.mc_transport_run(ctx, mc.make_lcg(), [W.to_mc_problem(p, mc)], mc.mc_run_config(precision=precision, **cfg), t.c)
        out.append((t.bins, t.counts, t.hist_state, t.hist_draws))
    for got in out[:-1]:
        for x, y in zip(got, out[-1]):
            assert torch.equal(x, y)
    ctx.close()
