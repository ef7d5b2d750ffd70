"""mc_lcg_draw_host into pageable buffers, or one pageable and one page-locked,
around the sizes at which page-locked ones are cut into slices: the device
call's states and digests, bit for bit, with seeds and with given states."""
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("pinned_states,pinned_digest", [(False, False), (True, False), (False, True)])
@pytest.mark.parametrize("n,draws", [(253_125, 64), (1_000_001, 64), (2**22 + 3, 2)])
@pytest.mark.parametrize("load", [False, True])
def test_matches_the_device_call(n, draws, pinned_states, pinned_digest, load):
    import torch

    import paper_2403_06362_gb300 as mc
    from paper_2403_06362_gb300 import workloads as W

    ctx, lcg = mc.Context(0), mc.make_lcg()
    spec = None if load else mc.mc_seed_spec(mode=mc.MC_SEED_HASH, seed=W.HASH_SEED)
    given = torch.arange(n, dtype=torch.int64) * 7919 + 5
    st, dg = given.cuda(), torch.empty(n, dtype=torch.int64, device="cuda")
    mc.mc_lcg_draw(ctx, lcg, spec, 9, st, n, draws, None, dg)
    h_st = given.pin_memory() if pinned_states else given.clone()
    h_dg = torch.zeros(n, dtype=torch.int64, pin_memory=pinned_digest)
    mc.mc_lcg_draw_host(ctx, lcg, spec, 9, h_st, n, draws, h_dg)
    assert torch.equal(h_st, st.cpu()) and torch.equal(h_dg, dg.cpu())
    only = torch.zeros(n, dtype=torch.int64, pin_memory=pinned_digest)
    if not load:  # digests alone
        mc.mc_lcg_draw_host(ctx, lcg, spec, 9, None, n, draws, only)
        assert torch.equal(only, dg.cpu())
    ctx.close()


@pytest.mark.parametrize("n", [2**19 - 1, 2**19])
def test_given_states_around_the_size_that_is_cut(n):
    import torch

    import paper_2403_06362_gb300 as mc

    ctx, lcg = mc.Context(0), mc.make_lcg()
    given = torch.arange(n, dtype=torch.int64) * 7919 + 5
    st, dg = given.cuda(), torch.empty(n, dtype=torch.int64, device="cuda")
    mc.mc_lcg_draw(ctx, lcg, None, 0, st, n, 100, None, dg)
    h_st, h_dg = given.pin_memory(), torch.zeros(n, dtype=torch.int64, pin_memory=True)
    mc.mc_lcg_draw_host(ctx, lcg, None, 0, h_st, n, 100, h_dg)
    assert torch.equal(h_st, st.cpu()) and torch.equal(h_dg, dg.cpu())
    ctx.close()
