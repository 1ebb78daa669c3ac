"""The segmented sweeps, the fused pre-smoothing residual + restriction and the
cluster's coarsest-level solve of the directed operator at the edges of the
shapes they are launched in: quads, pairs and single columns, ragged tiles,
layer counts around the segment lengths, more layers than a shape holds,
unaligned buffers.  Against the CPU oracle at the tolerances of the sweeps
(FP64 1e-12, FP32 2e-5) and of the V-cycles (FP64 1e-11; FP32 1e-4) elsewhere."""
import numpy as np
import pytest
import torch

from gpu_common import dev, host, rel_inf
from oracle import ns as N
from oracle import tpmg as O
from synthetic import make_ns_problem

pytestmark = pytest.mark.gpu

NAMES = ("h", "tx", "ty", "tz", "txr", "tyr", "tzr")


def handle(shape, seed, **params):
    from paper_2307_04528_gb300.solver import NSHandle
    P = make_ns_problem(*shape, 0.2, seed, pe=0.3)
    p = O.MGParams(**params)
    levels = N.build_hierarchy(*(P[k] for k in NAMES), p)
    return NSHandle(*(dev(P[k]) for k in NAMES), mixed=1, **params), levels, p


def scaled(levels, c):
    return [N.NSLevel(*(np.ascontiguousarray(a * c, dtype=np.float32) for a in lv.arrays()), lv.geo)
            for lv in levels]


def shifted(t):
    out = torch.empty(t.numel() + 1, dtype=t.dtype, device="cuda")[1:].view(t.shape)
    out.copy_(t)
    return out


SHAPES = [(132, 64, 5), (130, 66, 9), (129, 64, 11), (128, 64, 81),  # 8192 columns and more
          (64, 34, 37), (66, 32, 81), (64, 32, 33),                  # 2048 to 8191
          (30, 10, 1), (26, 14, 23), (5, 4, 73), (6, 4, 192)]


@pytest.mark.parametrize("shape", SHAPES, ids=lambda s: "x".join(map(str, s)))
def test_sweeps(shape):
    H, levels, p = handle(shape, sum(shape), levels=1)
    rng = np.random.default_rng(sum(shape))
    b, u = rng.standard_normal(levels[0].shape), rng.standard_normal(levels[0].shape)
    for tr, levs in ((False, levels), (True, N.transposed(levels))):
        for prec, lev, dt, tol in ((0, levs[0], torch.float64, 1e-12),
                                   (1, scaled(levs, H.fp32_scale)[0], torch.float32, 2e-5)):
            bb, uu = (a.astype(lev.h.dtype) for a in (b, u))
            zero = N.smooth_from_zero(lev, bb, p.omega)
            want = N.smooth(lev, bb, uu, p.omega)
            for put in (lambda a: dev(a, dt), lambda a: shifted(dev(a, dt))):
                got0 = H.level_smooth(0, put(bb), None, transpose=tr, prec=prec)
                got = H.level_smooth(0, put(bb), put(uu), transpose=tr, prec=prec)
                assert rel_inf(host(got0), zero) <= tol, (tr, prec)
                assert rel_inf(host(got), want) <= tol, (tr, prec)


# two levels each; the coarsest takes 2 to 12 layers per thread, or sweeps
@pytest.mark.parametrize("shape", [(8, 4, 3), (20, 12, 24), (36, 20, 37), (28, 12, 70),
                                   (16, 8, 100), (128, 66, 9)],
                         ids=lambda s: "x".join(map(str, s)))
def test_two_level_cycle(shape):
    H, levels, p = handle(shape, sum(shape), levels=2)
    r = np.random.default_rng(sum(shape)).standard_normal(levels[0].shape)
    for tr, levs in ((False, levels), (True, N.transposed(levels))):
        for prec, ls, dt, tol in ((0, levs, torch.float64, 1e-11),
                                  (1, scaled(levs, H.fp32_scale), torch.float32, 1e-4)):
            rr = r.astype(ls[0].h.dtype)
            want = N.vcycle(ls, rr, p)
            for t in (dev(rr, dt), shifted(dev(rr, dt))):
                assert rel_inf(host(H.vcycle(t, transpose=tr, prec=prec)), want) <= tol, (tr, prec)
