"""Replays of a captured slab launch of several problems whose processing
order differs in kind or in place from the captured call's: other sums of bin
counts behind the same launch shape, and a history range that ends where the
problems end in one call and before it in the next."""
import pytest

from paper_2403_06362_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def problems(bins, histories):
    out, off = [], 0
    for i, (b, n) in enumerate(zip(bins, histories)):
        out.append(W.slab_problem(10.0 + 20.0 * i, 1.0, 0.5 + 0.2 * i, n, b, 1, W.SEED_HASH_HIER, key=i,
                                  tally_offset=off))
        off += b
    return out


CALLS = {
    # the problems' counts agree in everything a launch's shape shows but the sum of their bins
    "bins": [((20, 5), (3000, 3000), 0), ((20, 20), (3000, 3000), 0), ((5, 20), (3000, 3000), 0),
             ((20, 5), (3000, 3000), 0)],
    "many_bins": [((64, 1, 1), (500, 700, 900), 0), ((64, 64, 64), (500, 700, 900), 0), ((1, 64, 1), (900, 700, 500), 0)],
    # 4000 histories each time: all of them, then the first 4000 of more
    "range": [((20, 20), (3000, 1000), 4000), ((20, 20), (3000, 2000), 4000), ((20, 20), (1000, 3000), 4000),
              ((20, 20), (4000, 1), 4000)],
}


@pytest.mark.parametrize("kind", sorted(CALLS))
def test_replays_equal_fresh_launches(kind):
    import torch

    import paper_2403_06362_gb300 as mc

    graphs, plain = mc.Context(0), mc.Context(0)
    # a larger call first: the record buffer keeps its place for all that follow
    n = len(CALLS[kind][0][0])
    big = [W.to_mc_problem(p, mc) for p in problems((200,) * n, (100,) * n)]
    t = mc.Tally(200 * n, n)
    mc.mc_transport_run(graphs, mc.make_lcg(), mc.problem_array(big), mc.mc_run_config(use_graph=1), t.c)
    torch.cuda.synchronize()
    for bins, histories, end in CALLS[kind]:
        arr = mc.problem_array([W.to_mc_problem(p, mc) for p in problems(bins, histories)])
        want = mc.Tally(200 * n, n)
        mc.mc_transport_run(graphs, mc.make_lcg(), arr, mc.mc_run_config(use_graph=1, range_end=end), t.c)
        mc.mc_transport_run(plain, mc.make_lcg(), arr, mc.mc_run_config(range_end=end), want.c)
        torch.cuda.synchronize()
        assert torch.equal(t.bins, want.bins) and torch.equal(t.counts, want.counts), (bins, histories, end)
    graphs.close()
    plain.close()
