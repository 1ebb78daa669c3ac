"""The FP64 stencil with a thread per 2 x 2 columns from the sizes (2^19 cells, or
2^20 below 16384 columns) at which the plain application and residual take it: one
layer, rows ending inside a warp, layers split between blocks; the CPU oracle at 1e-13,
and the same bits as the column walk or the cells' threads that a buffer one value off
alignment takes."""
import numpy as np
import pytest
import torch

from gpu_common import dev, handle_for, host, oracle_levels, problem, rel_inf
from oracle import tpmg as O

pytestmark = pytest.mark.gpu


def shifted(t):
    out = torch.empty(t.numel() + 1, dtype=t.dtype, device="cuda")[1:].view(t.shape)
    out.copy_(t)
    return out


@pytest.mark.parametrize("shape", [(130, 66, 124), (514, 256, 4), (1026, 512, 1), (128, 64, 128),
                                   (182, 92, 33), (128, 64, 127)],
                         ids=lambda s: "x".join(map(str, s)))
def test_stencil(shape):
    P = problem(*shape, sigma=0.2, seed=sum(shape))
    lev, _ = oracle_levels(P, levels=1)
    H = handle_for(P, levels=1, mixed=0)
    rng = np.random.default_rng(sum(shape))
    x, b = rng.standard_normal(lev[0].shape), rng.standard_normal(lev[0].shape)
    got, r = H.level_apply(0, dev(x)), H.level_residual(0, dev(b), dev(x))
    assert rel_inf(host(got), O.apply(lev[0], x)) <= 1e-13
    assert rel_inf(host(r), O.residual(lev[0], b, x)) <= 1e-13
    assert torch.equal(got, H.level_apply(0, shifted(dev(x))))
    assert torch.equal(r, H.level_residual(0, dev(b), shifted(dev(x))))
