"""The fp32-guarded transport keeps its bits: order-weighted checksums of the
int64 tallies of small box and slab runs, taken when the fp32 uniforms,
directions and distances were rounded from fp64 values by the fp64 unit.
(The fp32 path has no oracle; any other rounding of a draw, a distance or a
fixed-point length changes them.)"""
import numpy as np
import pytest

from paper_2403_06362_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def env():
    import paper_2403_06362_gb300 as mc
    ctx = mc.Context(0)
    yield mc, ctx
    ctx.close()


def checksum(tally):
    v = tally.bins.cpu().numpy().view(np.uint64).reshape(-1)
    with np.errstate(over="ignore"):
        return int((v * (2 * np.arange(v.size, dtype=np.uint64) + np.uint64(1))).sum(dtype=np.uint64))


@pytest.mark.parametrize("schedule", [0, 1])
@pytest.mark.parametrize("n,mesh,seeding,expected", [
    (5000, 16, W.SEED_HASH, 2473499926526575656),
    (20000, 50, W.SEED_STRIDE, 13858132224851247148)])
def test_box(env, schedule, n, mesh, seeding, expected):
    mc, ctx = env
    b = W.box_problem(n_histories=n, mesh=mesh, seeding=seeding)
    prob, spec = W.to_mc_box(b, mc)
    t = mc.Tally(W.box_tally_slots(b), 1)
    mc.mc_transport_run(ctx, mc.make_lcg(), mc.problem_array([prob]),
                        mc.mc_run_config(precision=mc.MC_FP32_GUARDED, schedule=schedule), t.c)
    assert checksum(t) == expected


@pytest.mark.parametrize("schedule", [0, 1])
@pytest.mark.parametrize("L,c,n,bins,seeding,expected", [
    (10.0, 0.5, 20000, 20, W.SEED_HASH, 9517234941280306),
    (200.0, 0.999, 3000, 200, W.SEED_STRIDE, 6411735516088348531),
    (2.0, 0.9, 5000, 7, W.SEED_HASH_HIER, 1147363928390249)])
def test_slab(env, schedule, L, c, n, bins, seeding, expected):
    mc, ctx = env
    p = [W.slab_problem(L, 1.0, c, n, bins, 3, seeding)]
    t = mc.Tally(W.tally_slots(p), 1)
    mc.mc_transport_run(ctx, mc.make_lcg(), [W.to_mc_problem(q, mc) for q in p],
                        mc.mc_run_config(precision=mc.MC_FP32_GUARDED, schedule=schedule), t.c)
    assert checksum(t) == expected
