"""Sweeps and coarsest-level solves of columns whose row sums fall or rise by a
large factor from one layer to the next, as at a jump of density or under
terrain: the vertical coupling is there a small part of the pivot below, and the
solution above hangs on its relative accuracy.  Against the CPU oracle at the
tolerances of the sweeps and coarse solves elsewhere (FP64 1e-13 and, for twelve
sweeps, 1e-12; Chebyshev 1e-11; FP32 2e-5)."""
import numpy as np
import pytest
import torch

from gpu_common import dev, handle_for, host, oracle_levels, rel_inf
from oracle import tpmg as O

pytestmark = pytest.mark.gpu


def contrast(nlon, nlat, nz, factor, coupling):
    """Fields with row sums of order 1 in the lower and 1 / factor in the upper
    half, vertical couplings `coupling` times the smaller of the two rows'."""
    rng = np.random.default_rng(nlon + nlat + nz)
    fac = np.where(np.arange(nz) < nz // 2, 1.0, 1.0 / factor)[:, None, None]
    draw = lambda: np.exp(0.1 * rng.standard_normal((nz, nlat, nlon)))
    h, tx, ty = fac * draw(), 0.2 * fac * draw(), 0.2 * fac * draw()
    ty[:, -1] = 0.0
    tz = np.zeros_like(h)
    tz[:-1] = coupling * np.minimum(fac[:-1], fac[1:]) * draw()[:-1]
    return dict(tx=tx, ty=ty, tz=tz, h=h), fac * rng.uniform(-1, 1, h.shape), \
        rng.uniform(-1, 1, h.shape)


SHAPES = [(30, 10, 16), (6, 4, 100), (64, 34, 70), (132, 64, 70), (128, 66, 37), (130, 64, 70),
          (129, 66, 12)]
# the last: the vertical coupling is the larger part of every pivot below the top
SYSTEMS = [(1e4, 0.1), (1e4, 10.0), (1e-4, 0.1), (1.0, 10.0)]


@pytest.mark.parametrize("factor,coupling", SYSTEMS)
@pytest.mark.parametrize("shape", SHAPES, ids=lambda s: "x".join(map(str, s)))
def test_sweeps(shape, factor, coupling):
    P, b, u = contrast(*shape, factor, coupling)
    lev, p = oracle_levels(P, levels=1)
    H = handle_for(P, levels=1)
    for prec, ol, dt, tol in ((0, lev[0], torch.float64, 1e-13),
                              (1, O.float_levels(lev)[0], torch.float32, 2e-5)):
        bb, uu = b.astype(ol.h.dtype), u.astype(ol.h.dtype)
        if prec:  # the FP32 operator is scaled by a power of two
            bb = bb * np.float32(H.fp32_scale)
        om = ol.h.dtype.type(p.omega)
        zero, guess = np.zeros_like(bb), uu.copy()
        O.smooth(ol, bb, zero, om)
        O.smooth(ol, bb, guess, om)
        tb, tu = dev(bb, dt), dev(uu, dt)
        assert rel_inf(host(H.level_smooth(0, tb, prec=prec)), zero) <= tol, prec
        assert rel_inf(host(H.level_smooth(0, tb, tu, prec=prec)), guess) <= tol, prec
        assert rel_inf(host(H.level_smooth_dot(0, tb, tu, prec=prec)[0]), guess) <= tol, prec


@pytest.mark.parametrize("factor,coupling", SYSTEMS)
@pytest.mark.parametrize("shape", [(8, 4, 16), (14, 6, 70), (10, 6, 100), (64, 34, 37)],
                         ids=lambda s: "x".join(map(str, s)))
def test_coarsest_solves(shape, factor, coupling):
    P, b, _ = contrast(*shape, factor, coupling)
    lev, p = oracle_levels(P, levels=1, coarse_method="chebyshev", coarse_iters=12)
    H = handle_for(P, levels=1, coarse_method=2, coarse_iters=12)
    for prec, ol, dt, tols in ((0, lev[0], torch.float64, (1e-12, 1e-11)),
                               (1, O.float_levels(lev)[0], torch.float32, (2e-5, 2e-5))):
        bb = b.astype(ol.h.dtype) * ol.h.dtype.type(H.fp32_scale if prec else 1.0)
        want = np.zeros_like(bb)
        for _ in range(12):
            O.smooth(ol, bb, want, ol.h.dtype.type(p.omega))
        tb = dev(bb, dt)
        assert rel_inf(host(H.level_relax(0, tb, 12, prec=prec)), want) <= tols[0], prec
        cheb = O.coarse_chebyshev(ol, bb, 12)
        assert rel_inf(host(H.coarse_solve(tb, prec=prec)), cheb) <= tols[1], prec
