"""The segmented sweeps at the edges of the shapes they are launched in: each
branch of the dispatch (quads, pairs and single columns; segments of 9, 5 and
3 layers; 8 to 64 columns to a block), ragged tiles, layer counts around a
multiple of the segment length, more layers than the shapes hold, unaligned
buffers, and the one-block coarsest-level solve for each of its segment
lengths.  Against the CPU oracle, FP64 1e-13 and FP32 2e-5 in the max norm (the
sweep's tolerances elsewhere; 12 sweeps: 1e-12 and 2e-5)."""
import numpy as np
import pytest
import torch

from gpu_common import dev, handle_for, host, oracle_levels, problem, rel_inf
from oracle import tpmg as O

pytestmark = pytest.mark.gpu

# nlon, nlat, nz: one level each
SHAPES = [
    (132, 64, 9), (132, 64, 10), (128, 64, 72),   # quads, 9 layers per segment
    (128, 66, 37), (100, 90, 5),                  # quads, 5 layers per segment
    (130, 66, 9), (129, 64, 20),                  # pairs / single columns from zero, walk on a guess
    (128, 64, 73),                                # more layers than the shapes: the walk
    (64, 34, 37), (66, 32, 80), (66, 32, 81),     # 2048 to 8191 columns
    (30, 10, 1), (26, 14, 23), (5, 4, 73), (6, 4, 192),  # small levels
]


@pytest.mark.parametrize("shape", SHAPES, ids=lambda s: "x".join(map(str, s)))
def test_sweeps(shape):
    P = problem(*shape, sigma=0.2, seed=sum(shape))
    lev, p = oracle_levels(P, levels=1)
    H = handle_for(P, levels=1)
    rng = np.random.default_rng(sum(shape) + 1)
    b = rng.standard_normal(lev[0].shape)
    u = rng.standard_normal(lev[0].shape)
    for prec, ol, dt, tol in ((0, lev[0], np.float64, 1e-13),
                              (1, O.float_levels(lev)[0], np.float32, 2e-5)):
        om = dt(p.omega)
        bb, uu = b.astype(dt), u.astype(dt)
        tb, tu = (dev(a, torch.float64 if prec == 0 else torch.float32) for a in (bb, uu))
        ref0, ref = np.zeros_like(bb), uu.copy()
        O.smooth(ol, bb, ref0, om)
        O.smooth(ol, bb, ref, om)
        assert rel_inf(host(H.level_smooth(0, tb, prec=prec)), ref0) <= tol
        assert rel_inf(host(H.level_smooth(0, tb, tu, prec=prec)), ref) <= tol
        got, dot = H.level_smooth_dot(0, tb, tu, prec=prec)
        assert rel_inf(host(got), ref) <= tol
        assert abs(dot - O.dot(bb, ref)) <= tol * O.norm2(bb) * O.norm2(ref)
        # buffers one value off alignment
        n = bb.size
        buf = torch.empty(2 * n + 1, dtype=tb.dtype, device="cuda")
        ob, ou = buf[1:n + 1].view(tb.shape), buf[n + 1:].view(tb.shape)
        ob.copy_(tb)
        ou.copy_(tu)
        assert rel_inf(host(H.level_smooth(0, ob, ou, prec=prec)), ref) <= tol


# cells and columns that take 2, 4, 6, 8, 12 and 16 layers per thread, FP64's
# bound of 512 cells and one past FP32's of 8192
@pytest.mark.parametrize("shape", [(8, 4, 16), (14, 6, 24), (14, 6, 70), (18, 10, 37),
                                   (16, 14, 30), (32, 16, 16), (32, 20, 12), (16, 16, 33)],
                         ids=lambda s: "x".join(map(str, s)))
@pytest.mark.parametrize("sweeps", [1, 12])
def test_coarsest_solve(shape, sweeps):
    P = problem(*shape, sigma=0.2, seed=sum(shape))
    lev, p = oracle_levels(P, levels=1)
    H = handle_for(P, levels=1)
    b = np.random.default_rng(sum(shape)).standard_normal(lev[0].shape)
    for prec, ol, dt, tol in ((0, lev[0], np.float64, 1e-12),
                              (1, O.float_levels(lev)[0], np.float32, 2e-5)):
        bb = b.astype(dt)
        ref = np.zeros_like(bb)
        for _ in range(sweeps):
            O.smooth(ol, bb, ref, dt(p.omega))
        tb = dev(bb, torch.float64 if prec == 0 else torch.float32)
        assert rel_inf(host(H.level_relax(0, tb, sweeps, prec=prec)), ref) <= tol
