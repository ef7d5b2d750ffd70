"""A slab run captured by the caller and replayed between other runs of its
context: the replay writes its own problem records, and a run whose records
were the last ones uploaded must not take them for its own."""
import pytest

from paper_2403_06362_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def test_runs_around_a_replay():
    import torch

    import paper_2403_06362_gb300 as mc

    ctx, plain = mc.Context(0), mc.Context(0)
    lcg = mc.make_lcg()
    few = W.slab_batched(W.SEED_HASH_HIER, n_problems=5, max_histories=2000, n_bins=20, seed=3)
    many = W.slab_batched(W.SEED_HASH_HIER, n_problems=17, max_histories=2000, n_bins=20, seed=4)
    arrays = [mc.problem_array([W.to_mc_problem(p, mc) for p in probs]) for probs in (few, many)]
    tallies = [mc.Tally(17 * 20, n) for n in (5, 17)]
    want = []
    for arr, n in zip(arrays, (5, 17)):
        t = mc.Tally(17 * 20, n)
        mc.mc_transport_run(plain, lcg, arr, mc.mc_run_config(), t.c)
        want.append(t)

    def check(i):
        torch.cuda.synchronize()
        assert torch.equal(tallies[i].bins, want[i].bins) and torch.equal(tallies[i].counts, want[i].counts)
        tallies[i].bins.fill_(-1)
        tallies[i].counts.fill_(-1)

    for i in (1, 0):  # the buffers get their size
        mc.mc_transport_run(ctx, lcg, arrays[i], mc.mc_run_config(), tallies[i].c)
        check(i)
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        mc.mc_transport_run(ctx, lcg, arrays[0], mc.mc_run_config(), tallies[0].c)
    for _ in range(2):
        mc.mc_transport_run(ctx, lcg, arrays[1], mc.mc_run_config(), tallies[1].c)
        check(1)
        graph.replay()
        check(0)
        mc.mc_transport_run(ctx, lcg, arrays[1], mc.mc_run_config(), tallies[1].c)
        check(1)
    del graph
    ctx.close()
    plain.close()
