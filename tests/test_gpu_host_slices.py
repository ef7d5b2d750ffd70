"""mc_lcg_draw_host over the sizes at which its number of slices changes: the
device call's states and digests, bit for bit."""
import pytest

pytestmark = pytest.mark.gpu


# 64 draws: two slices from 253 125 streams on; 129 draws: one slice; 33
# draws: the smallest slice; 1 draw: more than the largest slice.
@pytest.mark.parametrize("n,draws", [(253_124, 64), (253_125, 64), (262_145, 64), (1_000_001, 64), (700_000, 129),
                                     (500_000, 33), (2**22 + 1, 1)])
def test_slices_match_the_device_call(n, draws):
    import torch

    import paper_2403_06362_gb300 as mc
    from paper_2403_06362_gb300 import workloads as W

    ctx, lcg = mc.Context(0), mc.make_lcg()
    spec = mc.mc_seed_spec(mode=mc.MC_SEED_STRIDE, seed=W.STRIDE_X0, stride_q=W.STRIDE_Q)
    st = torch.empty(n, dtype=torch.int64, device="cuda")
    dg = torch.empty_like(st)
    mc.mc_lcg_draw(ctx, lcg, spec, 9, st, n, draws, None, dg)
    h_st = torch.empty(n, dtype=torch.int64, pin_memory=True)
    h_dg = torch.empty(n, dtype=torch.int64, pin_memory=True)
    mc.mc_lcg_draw_host(ctx, lcg, spec, 9, h_st, n, draws, h_dg)
    assert torch.equal(h_st, st.cpu()) and torch.equal(h_dg, dg.cpu())
    ctx.close()
