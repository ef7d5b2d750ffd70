"""The slab history kernel at the edges of its bin walk and its counters: one
bin, bins far narrower and far wider than a flight, more bins than the shared
tables hold, a beam (first flight from an edge), histories that nearly all
exceed the stride, several problems in a launch; against the oracle, and
between the schedules and precisions that keep no bin between flights."""
import numpy as np
import pytest

from paper_2403_06362_gb300 import workloads as W
from paper_2403_06362_gb300._ffi import MC_NCOUNT

pytestmark = pytest.mark.gpu

TOL = 1e-6  # the parity bar of the slab tallies: the oracle's logarithm may differ by one ulp


@pytest.fixture(scope="module")
def env():
    import torch
    import paper_2403_06362_gb300 as mc
    ctx = mc.Context(0)
    yield mc, ctx, torch
    torch.cuda.synchronize()
    ctx.close()


def run(env, probs, **cfg):
    mc, ctx, torch = env
    n = sum(p["n_histories"] for p in probs)
    t = mc.Tally(W.tally_slots(probs), len(probs), n_histories=n)
    mc.mc_transport_run(ctx, mc.make_lcg(), [W.to_mc_problem(p, mc) for p in probs], mc.mc_run_config(**cfg), t.c)
    torch.cuda.synchronize()
    return (t.bins.cpu().numpy(), t.counts.cpu().numpy().view(np.uint64).reshape(-1, MC_NCOUNT),
            t.hist_state.cpu().numpy().view(np.uint64), t.hist_draws.cpu().numpy().view(np.uint64))


def problem(bins, L=10.0, sigma_t=1.0, c=0.8, source=W.SRC_ISOTROPIC, q=W.STRIDE_Q, seeding=W.SEED_HASH, n=2001, **kw):
    return W.slab_problem(L, sigma_t, c, n, bins, 3, seeding, source=source, stride_q=q, **kw)


CASES = [problem(1), problem(2, c=0.99), problem(7, L=0.3), problem(64, L=200.0, c=0.99), problem(4095), problem(5000, n=301),
         problem(33, source=W.SRC_BEAM), problem(20, L=1e-3, c=1.0, source=W.SRC_BEAM),
         problem(20, q=4, seeding=W.SEED_STRIDE, c=0.95)]


@pytest.mark.parametrize("i", range(len(CASES)))
def test_against_the_oracle(env, oracle, i):
    p = CASES[i]
    bins, counts, state, draws = run(env, [p])
    o = oracle.slab_run(oracle.Lcg(m=63, pad=0, g=W.LCG_G, c=1), W.to_oracle_problem(p, oracle), per_history=True)
    assert np.array_equal(state, o["hist_state"]) and np.array_equal(draws, o["hist_draws"])
    oc = np.asarray(o["counts"], dtype=np.uint64)
    k = min(len(oc), 14)
    assert np.array_equal(counts[0, :k], oc[:k])
    exp = o["tally"].astype(np.float64).reshape(-1)
    assert np.all(np.abs(bins - exp) <= TOL * np.abs(exp))


@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("i", range(len(CASES)))
def test_schedules_and_shapes_agree(env, i, precision):
    ref = run(env, [CASES[i]], precision=precision)
    for cfg in (dict(schedule=1), dict(block=32, chunk=3), dict(block=512, tally_mode=2), dict(tally_atomics=2)):
        got = run(env, [CASES[i]], precision=precision, **cfg)
        for x, y in zip(ref, got):
            assert np.array_equal(x, y), cfg


def test_exceedances_of_several_problems(env):
    probs, off, ids = [], 0, 0
    for i in range(5):
        p = problem(5 + i, q=3 + i, seeding=W.SEED_STRIDE, c=0.9, n=500 + i, tally_offset=off, id_offset=ids)
        off += p["n_bins"] * p["n_batches"]
        ids += p["n_histories"]
        probs.append(p)
    together = run(env, probs)
    one = [run(env, [dict(p, tally_offset=0)]) for p in probs]
    assert np.array_equal(together[0], np.concatenate([r[0] for r in one]))
    assert np.array_equal(together[1], np.concatenate([r[1] for r in one]))
    assert np.all(together[1][:, 8] > 0)


@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("block", [64, 96, 160, 256, 512])
def test_cooperative_tail_of_any_block(env, block, precision):
    """Long chains of several problems through the tail (blocks of 64 threads
    and more), with and without row caches, against single-warp blocks, which
    have none."""
    probs, off = [], 0
    for i, (bins, batches) in enumerate([(7, 3), (200, 20), (300, 20)]):
        probs.append(W.slab_problem(60.0, 1.0, 0.999, 150, bins, batches, W.SEED_HASH_HIER, key=i, tally_offset=off))
        off += bins * batches
    for some in (probs, probs[:2]):  # with 300 bins no row is cached
        ref = run(env, some, precision=precision, block=32)
        for cfg in (dict(), dict(tally_mode=2), dict(blocks_per_sm=1, chunk=8), dict(event_cap=40)):
            want = ref if "event_cap" not in cfg else run(env, some, precision=precision, block=32, **cfg)
            got = run(env, some, precision=precision, block=block, **cfg)
            for x, y in zip(want, got):
                assert np.array_equal(x, y), cfg
