"""The fused residual + restriction for each height of its bands against the residual
and the restriction as kernels of their own: the same bits."""
import pytest
import torch

from gpu_common import handle_for, problem

pytestmark = pytest.mark.gpu


# FP64 in full and after one sweep: bands of 1, 2, 4, 8 and 16 coarse rows; rows of
# several warps and of one, odd layers
@pytest.mark.parametrize("shape", [(8, 4, 3), (64, 32, 16), (128, 96, 40), (132, 66, 71),
                                   (256, 192, 70), (384, 256, 50), (1024, 768, 16)],
                         ids=lambda s: "x".join(map(str, s)))
def test_bands(shape):
    H = handle_for(problem(*shape, sigma=0.2, seed=sum(shape)), levels=2, mixed=0)
    gen = torch.Generator(device="cuda").manual_seed(7)
    b, u = (torch.randn(shape[::-1], generator=gen, device="cuda", dtype=torch.float64)
            for _ in range(2))
    want = H.level_restrict(0, H.level_residual(0, b, u))
    assert torch.equal(H.level_residual_restrict(0, b, u), want)
    # u of one sweep from zero: its residual by the couplings alone, to rounding
    s = H.level_smooth(0, b)
    full = H.level_residual_restrict(0, b, s)
    pre = H.level_presmooth_restrict(0, b, s)
    assert torch.max(torch.abs(pre - full)) <= 1e-10 * torch.max(torch.abs(b))
