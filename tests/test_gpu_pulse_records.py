"""Families of the pulse kernels at the edges of their records: fewer sources
than a warp has lanes, so that records are given away from the start; stacks of
a few entries, whose ring wraps and overflows meanwhile; collisions of up to
eight and of thirty secondaries, so that one record holds more than the stack.
Per-history states and draw counts, counters and tallies against the oracle
(whose stack is unbounded); a run's results do not depend on who follows a
family, so a second run gives the same."""
import numpy as np
import pytest

from paper_2403_06362_gb300 import workloads as W
from paper_2403_06362_gb300._ffi import MC_NCOUNT

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def env():
    import torch
    import paper_2403_06362_gb300 as mc
    ctx = mc.Context(0)
    yield mc, ctx, torch
    torch.cuda.synchronize()
    ctx.close()


def run(env, a, **cfg):
    mc, ctx, torch = env
    prob, spec = W.to_mc_pulse(a, mc)
    n = W.azurv1_histories(a) if a["n_census"] < 2 else 0
    t = mc.Tally(W.azurv1_tally_slots(a), 1, n_histories=n)
    mc.mc_transport_run(ctx, mc.make_lcg(), mc.problem_array([prob]), mc.mc_run_config(**cfg), t.c)
    torch.cuda.synchronize()
    counts = t.counts.cpu().numpy().view(np.uint64).reshape(-1, MC_NCOUNT)[0]
    per = [v.cpu().numpy().view(np.uint64) for v in (t.hist_state, t.hist_draws)] if n else []
    return [t.bins.cpu().numpy().view(np.int64), counts] + per


def problem(seeding, sources, c, nu, t_end, n_batches=1, **kw):
    return W.azurv1(seeding=seeding, n_reps=1, n_batches=n_batches, per_batch=sources, c=c, nu=nu, t_end=float(t_end),
                    n_time_bins=t_end, seed=3, **kw)


def lcg(oracle):
    return oracle.Lcg(m=63, pad=0, g=W.LCG_G, c=1)


@pytest.mark.parametrize("depth", [1, 2, 3, 5, 16, 0])
@pytest.mark.parametrize("sources,c,nu,t_end", [(1, 0.9, 1.3, 40), (20, 0.2, 8.0, 8), (33, 0.07, 30.0, 6),
                                                (33, 0.25, 5.0, 16), (70, 0.4, 2.75, 20)])
def test_hash_families(env, oracle, sources, c, nu, t_end, depth):
    a = problem(W.SEED_HASH_HIER, sources, c, nu, t_end)
    o = oracle.azurv1_run(lcg(oracle), W.to_oracle_azurv1(a, oracle), per_history=True)
    for cfg in (dict(stack_depth=depth), dict(stack_depth=depth), dict(stack_depth=depth, block=64, tally_atomics=2)):
        bins, counts, state, draws = run(env, a, **cfg)
        assert np.array_equal(state, o["hist_state"]) and np.array_equal(draws, o["hist_draws"]), cfg
        assert np.array_equal(counts[:15], o["counts"][:15]) and counts[15] == 0, cfg
        assert np.array_equal(bins, o["tally"]), cfg


@pytest.mark.parametrize("sources,c,nu,t_end", [(1, 0.9, 1.3, 20), (20, 0.2, 8.0, 8), (33, 0.25, 5.0, 16),
                                                (70, 0.4, 2.75, 20), (3, 1.0, 1.0, 20)])
def test_stride_families(env, oracle, sources, c, nu, t_end):
    a = problem(W.SEED_STRIDE, sources, c, nu, t_end)
    o = oracle.azurv1_run(lcg(oracle), W.to_oracle_azurv1(a, oracle), per_history=True)
    for cfg in (dict(), dict(block=64, tally_atomics=2), dict(chunk=3)):
        bins, counts, state, draws = run(env, a, **cfg)
        assert np.array_equal(state, o["hist_state"]) and np.array_equal(draws, o["hist_draws"]), cfg
        assert np.array_equal(counts[:15], o["counts"][:15]) and counts[15] == 0, cfg
        assert np.array_equal(bins, o["tally"]), cfg


@pytest.mark.parametrize("depth", [1, 3, 16, 0])
@pytest.mark.parametrize("sources,c,nu,t_end", [(20, 0.2, 8.0, 8), (33, 0.25, 5.0, 16), (70, 0.4, 2.75, 20)])
def test_census_families(env, oracle, sources, c, nu, t_end, depth):
    a = problem(W.SEED_HASH_HIER, sources, c, nu, t_end, n_batches=3, n_census=3)
    o = oracle.azurv1_census_run(lcg(oracle), W.to_oracle_azurv1(a, oracle))
    bins, counts = run(env, a, stack_depth=depth)
    assert np.array_equal(bins, np.asarray(o["tally"]).reshape(-1))
    assert np.array_equal(counts[:15], np.asarray(o["counts"], dtype=np.uint64)[:15]) and counts[15] == 0
