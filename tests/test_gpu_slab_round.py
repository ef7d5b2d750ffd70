"""A slab piece's fixed point is rounded by an addition below 2^51 and from its
bits above: pieces on both sides of that (2^51 / 2^32 = 524288 cm), and the
event schedule, which rounds all of them from the bits, give the same sums."""
import numpy as np
import pytest

from paper_2403_06362_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("bins", [1, 3, 40, 300])
@pytest.mark.parametrize("thick", [1e5, 1048576.0, 3e7])
def test_long_pieces(bins, thick):
    import torch

    import paper_2403_06362_gb300 as mc

    # 101 histories of a few flights, 10^6 cm each on the mean: some 10^9 cm, 4e18
    # in fixed point, below 2^63
    p = W.slab_problem(thick, 10.0 / thick, 0.5, 101, bins, 1, W.SEED_HASH)
    ctx, got = mc.Context(0), []
    for cfg in (dict(), dict(tally_mode=2, block=64), dict(schedule=1)):
        t = mc.Tally(W.tally_slots([p]), 1)
        mc.mc_transport_run(ctx, mc.make_lcg(), [W.to_mc_problem(p, mc)], mc.mc_run_config(**cfg), t.c)
        torch.cuda.synchronize()
        got.append(t.bins.cpu().numpy())
    assert got[0].sum() > 0
    for g in got[1:]:
        assert np.array_equal(got[0], g)
