"""Runs of one context whose problem records are, or are not, those of the call
before: repeated, changed in one field, of another count, another geometry or
another tally size in between, accumulated, replayed by the library's own
graph. Each against the same call under a context of its own."""
import pytest

from paper_2403_06362_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def slabs(n, bins, seed, c=0.7):
    return [W.slab_problem(8.0 + i, 1.0, c, 700 + i, bins, 2, W.SEED_HASH_HIER, key=i, seed=seed, tally_offset=2 * bins * i)
            for i in range(n)]


def test_each_call_is_as_under_a_fresh_context():
    import torch

    import paper_2403_06362_gb300 as mc

    lcg, slots = mc.make_lcg(), 1 << 15
    box, spec = W.to_mc_box(W.box_problem(n_histories=500, mesh=8), mc)
    a, b = slabs(1, 20, 1), slabs(1, 20, 2)
    many, wide = slabs(17, 20, 1), slabs(2, 4000, 3)
    calls = [(a, {}), (a, {}), (b, {}), (a, {}), (a, dict(schedule=1)), (a, dict(accumulate=1)), (a, dict(use_graph=1)),
             (a, {}), ([box], {}), (a, {}), (many, {}), (many, {}), (a, {}), (wide, {}), (wide, {}), (wide, dict(schedule=1)),
             (wide, dict(tally_mode=2)), (slabs(1, 3500, 4), {}), (slabs(1, 3500, 4), dict(schedule=1)), (a, dict(big=1)),
             (a, {}), (slabs(1, 20, 1, c=0.8), {}), (a, dict(precision=1)), (a, dict(range_end=0, range_begin=5))]
    ctx = mc.Context(0)
    for i, (probs, kw) in enumerate(calls):
        kw = dict(kw)
        n = (1 << 19) + 8 if kw.pop("big", 0) else slots
        arr = mc.problem_array([p if not isinstance(p, dict) else W.to_mc_problem(p, mc) for p in probs])
        got, want = mc.Tally(n, len(probs)), mc.Tally(n, len(probs))
        for t in (got, want):
            t.bins.fill_(7)
            t.counts.fill_(7)
        mc.mc_transport_run(ctx, lcg, arr, mc.mc_run_config(**kw), got.c)
        fresh = mc.Context(0)
        mc.mc_transport_run(fresh, lcg, arr, mc.mc_run_config(**kw), want.c)
        torch.cuda.synchronize()
        assert torch.equal(got.bins, want.bins) and torch.equal(got.counts, want.counts), i
        fresh.close()
    ctx.close()
