"""The box history kernel where its parts meet: meshes whose planes coincide
with the box faces or fall outside the shared plane table's usual size, runs
smaller than a warp or a refill, several problems in one launch (block
counters in shared memory and, beyond 16 problems, straight to the caller's),
every block size, against the oracle and against one-problem launches."""
import numpy as np
import pytest

from paper_2403_06362_gb300 import workloads as W
from paper_2403_06362_gb300._ffi import MC_NCOUNT

pytestmark = pytest.mark.gpu

TOL = 1e-6  # the parity bar of the box tallies: the oracle's logarithm may differ by one ulp


@pytest.fixture(scope="module")
def env():
    import torch
    import paper_2403_06362_gb300 as mc
    ctx = mc.Context(0)
    yield mc, ctx, torch
    torch.cuda.synchronize()
    ctx.close()


def run(env, boxes, **cfg):
    """One launch over the boxes (tally offsets and global ids in order)."""
    mc, ctx, torch = env
    probs, specs, off = [], [], 0
    for b in boxes:
        b["tally_offset"] = off
        p, s = W.to_mc_box(b, mc)
        probs.append(p)
        specs.append(s)
        off = W.box_tally_slots(b)
    n = sum(b["n_histories"] for b in boxes)
    t = mc.Tally(off, len(boxes), n_histories=n)
    mc.mc_transport_run(ctx, mc.make_lcg(), mc.problem_array(probs), mc.mc_run_config(**cfg), t.c)
    torch.cuda.synchronize()
    return (t.bins.cpu().numpy(), t.counts.cpu().numpy().view(np.uint64).reshape(-1, MC_NCOUNT),
            t.hist_state.cpu().numpy().view(np.uint64), t.hist_draws.cpu().numpy().view(np.uint64))


@pytest.mark.parametrize("mesh", [1, 2, 10, 37, 129])
@pytest.mark.parametrize("n,batches,seeding", [(1, 1, W.SEED_HASH), (33, 3, W.SEED_STRIDE), (1500, 7, W.SEED_HASH_HIER)])
def test_meshes_and_small_runs_match_the_oracle(env, oracle, mesh, n, batches, seeding):
    b = W.box_problem(n_histories=n, mesh=mesh, n_batches=batches, seeding=seeding)
    bins, counts, state, draws = run(env, [b])
    o = oracle.box_run(oracle.Lcg(m=63, pad=0, g=W.LCG_G, c=1), W.to_oracle_box(b, oracle), per_history=True)
    assert np.array_equal(state, o["hist_state"]) and np.array_equal(draws, o["hist_draws"])
    assert np.array_equal(counts[0, :15], o["counts"][:15])
    exp = o["tally"].astype(np.float64)
    assert np.all(np.abs(bins - exp) <= TOL * np.abs(exp))


@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("problems", [2, 17])
def test_several_problems_in_one_launch(env, problems, precision):
    def boxes():
        return [W.box_problem(n_histories=101 + 7 * i, mesh=4 + i, c=(0.5 + 0.02 * i, 0.3), seed=5 + i)
                for i in range(problems)]
    bins, counts, state, draws = run(env, boxes(), precision=precision)
    one = [run(env, [b], precision=precision) for b in boxes()]
    assert np.array_equal(bins, np.concatenate([r[0] for r in one]))
    assert np.array_equal(counts, np.concatenate([r[1] for r in one]))
    assert np.array_equal(state, np.concatenate([r[2] for r in one]))
    assert np.array_equal(draws, np.concatenate([r[3] for r in one]))


@pytest.mark.parametrize("precision", [0, 1])
def test_launch_shapes_and_schedules_agree(env, precision):
    ref = run(env, [W.box_problem(n_histories=3001, mesh=16)], precision=precision)
    for cfg in (dict(block=32, chunk=1), dict(block=96, chunk=5), dict(block=256, chunk=1000, blocks_per_sm=1),
                dict(tally_atomics=2), dict(schedule=1)):
        got = run(env, [W.box_problem(n_histories=3001, mesh=16)], precision=precision, **cfg)
        for x, y in zip(ref, got):
            assert np.array_equal(x, y), cfg


@pytest.mark.parametrize("side,inner", [
    (50.0, (0.0, 20.0)),           # the cube in a corner: entry and exit faces coincide
    (10.0, (0.0, 10.0)),           # the cube fills the box
    (50.0, (49.999, 50.0)),        # a sliver
    (80.0, (39.9999999, 40.0)),
    (2.0**-45, (2.0**-47, 2.0**-46)),  # outside the range of the fp32 decisions
    (2.0**45, (2.0**43, 2.0**44))])
def test_geometries_match_the_oracle(env, oracle, side, inner):
    """fp64 decides its faces in fp32 where that is sure; every form of the
    geometry, and the window's roulette, against the oracle."""
    b = W.box_problem(n_histories=3000, mesh=8, side=side, inner=inner, sigma_t=(25.0 / side, 60.0 / side))
    bins, counts, state, draws = run(env, [b])
    o = oracle.box_run(oracle.Lcg(m=63, pad=0, g=W.LCG_G, c=1), W.to_oracle_box(b, oracle), per_history=True)
    assert np.array_equal(state, o["hist_state"]) and np.array_equal(draws, o["hist_draws"])
    assert np.array_equal(counts[0, :15], o["counts"][:15])
    if side >= 2.0**20:
        return  # 3000 histories' tracks leave the int64 fixed point (2^-32 cm): no tally is defined
    # int64 fixed point of a track is off by at most one unit per contribution
    exp = o["tally"].astype(np.float64)
    assert np.all(np.abs(bins - exp) <= TOL * np.abs(exp) + counts[0, 1])
