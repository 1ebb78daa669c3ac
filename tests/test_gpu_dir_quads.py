"""The FP32 direction update + apply with a thread per four columns at the edges
of its tiles: the smallest rows, rows ending inside a warp, one layer, and layer
ranges split between blocks; every value equal, bit for bit, to the column walk
that a buffer one value off alignment takes, and to the oracle at the stencil's
FP32 tolerance (2e-5)."""
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


@pytest.mark.parametrize("shape", [(4, 2, 1), (4, 2, 3), (8, 4, 73), (20, 6, 9), (132, 10, 33),
                                   (260, 66, 16), (6, 4, 3)], ids=lambda s: "x".join(map(str, s)))
@pytest.mark.parametrize("beta", [None, 0.37])
def test_dir_apply(shape, beta):
    P = problem(*shape, sigma=0.2, seed=sum(shape))
    lev, _ = oracle_levels(P, levels=1)
    f = O.float_levels(lev)[0]
    H = handle_for(P, levels=1)
    rng = np.random.default_rng(sum(shape))
    z = dev(rng.standard_normal(f.shape), torch.float32)
    d = dev(rng.standard_normal(f.shape), torch.float32) if beta else None
    dn, q, dot = H.level_dir_apply(0, z, d, beta or 0.0, prec=1)
    dn2, q2, dot2 = H.level_dir_apply(0, shifted(z), None if d is None else shifted(d),
                                      beta or 0.0, prec=1)
    assert torch.equal(dn, dn2) and torch.equal(q, q2)
    assert rel_inf(host(q), O.apply(f, host(dn))) <= 2e-5
    scale = O.norm2(host(dn)) * O.norm2(host(q))
    assert abs(dot - dot2) <= 1e-6 * scale
    assert abs(dot - O.dot(host(dn), host(q))) <= 1e-5 * scale
