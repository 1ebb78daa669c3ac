"""The Chebyshev coarsest-level solve, one launch per step, against the CPU oracle
at the tolerances of the coarse solves elsewhere (FP64 1e-11, FP32 2e-5)."""
import numpy as np
import pytest
import torch

from gpu_common import dev, handle_for, host, oracle_levels, problem, rel_inf
from oracle import tpmg as O

pytestmark = pytest.mark.gpu


def check(shape, steps):
    P = problem(*shape, sigma=0.2, seed=sum(shape))
    lev, p = oracle_levels(P, levels=1, coarse_method="chebyshev", coarse_iters=steps)
    H = handle_for(P, levels=1, coarse_method=2, coarse_iters=steps)
    b = np.random.default_rng(sum(shape) + steps).standard_normal(lev[0].shape)
    for prec, ol, dt, tol in ((0, lev[0], torch.float64, 1e-11),
                              (1, O.float_levels(lev)[0], torch.float32, 2e-5)):
        bb = b.astype(ol.h.dtype)
        want = O.coarse_chebyshev(ol, bb, steps)
        tb = dev(bb, dt)
        off = torch.empty(tb.numel() + 1, dtype=dt, device="cuda")[1:].view(tb.shape)
        off.copy_(tb)
        for t in (tb, off):
            assert rel_inf(host(H.coarse_solve(t, prec=prec)), want) <= tol, prec


# one layer: the warp's other segments hold none, nor has theirs one below
@pytest.mark.parametrize("shape", [(8, 4, 1), (64, 34, 1), (128, 64, 1)],
                         ids=lambda s: "x".join(map(str, s)))
def test_one_layer(shape):
    check(shape, 5)


# The shapes of a step, whose residual has two copies, written in turn: pairs and
# 9-layer segments of single columns, quads in segments of 9 and 5, ragged tiles and
# last segments, single columns, more than 72 layers, and sizes that take the
# separate kernels.
@pytest.mark.parametrize("steps", [2, 3, 7, 24])
@pytest.mark.parametrize("shape", [(64, 34, 37), (64, 98, 70), (132, 64, 10), (128, 66, 37),
                                   (65, 34, 12), (6, 4, 100), (10, 6, 2), (129, 64, 9)],
                         ids=lambda s: "x".join(map(str, s)))
def test_steps(shape, steps):
    check(shape, steps)
