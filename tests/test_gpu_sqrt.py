"""The integer-pipe square root on the device, which starts from another
estimate than the host copy that tests/test_sqrt_exact.py checks: the same
bits as CUDA's correctly rounded sqrt over the direction sampler's arguments
1 - s, every mantissa pattern at even and odd exponents, and the neighbours of
exact squares, where the rounding is closest to a tie."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

N = 1 << 21


def arguments(kind):
    rng = np.random.default_rng(2403)
    if kind == "direction":  # 1 - s for s = v1^2 + v2^2 < 1, rounded as the sampler rounds it
        v = 2.0 * (rng.integers(0, 2**53, size=(2, 2 * N)) * 2.0**-53) - 1.0
        s = v[0] * v[0] + v[1] * v[1]
        return (1.0 - s[s < 1.0])[:N]
    if kind == "exponents":
        e = rng.integers(1, 2047, size=N, dtype=np.uint64)
        return ((e << np.uint64(52)) | rng.integers(0, 2**52, size=N, dtype=np.uint64)).view(np.float64)
    if kind == "squares":
        y = rng.integers(2**26, 2**27, size=N).astype(np.float64) * 2.0**-27
        b = (y * y).view(np.uint64) + rng.integers(0, 5, size=N, dtype=np.uint64) - np.uint64(2)
        return b.view(np.float64)
    m = np.concatenate([np.arange(4096), 2**52 - 1 - np.arange(4096), 2**np.arange(52), 2**52 - 2**np.arange(52)])
    e = np.arange(1000, 1047)
    return ((e[:, None].astype(np.uint64) << np.uint64(52)) | m[None, :].astype(np.uint64)).reshape(-1).view(np.float64)


@pytest.mark.parametrize("kind", ["direction", "exponents", "squares", "edges"])
def test_device_square_root_matches_cuda(kind):
    import torch

    import paper_2403_06362_gb300 as mc

    x = arguments(kind)
    dx = torch.from_numpy(x).cuda()
    ours, lib = torch.empty_like(dx), torch.empty_like(dx)
    mc.mc_sqrt_rn_device(dx, ours, 0)
    mc.mc_sqrt_rn_device(dx, lib, 1)
    torch.cuda.synchronize()
    ours, lib = ours.cpu().numpy(), lib.cpu().numpy()
    assert np.array_equal(lib.view(np.uint64), np.sqrt(x).view(np.uint64))
    assert np.array_equal(ours.view(np.uint64), lib.view(np.uint64))
