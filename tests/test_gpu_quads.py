"""The FP64 stencil with a thread per 2 x 2 columns and the prolongation with
a thread per four cells, at the edges of their tiles: the smallest grid, rows
that end inside a warp, a layer range split between blocks, and sizes and
buffers that take the general kernels instead.  Against the CPU oracles at the
tolerances of the stencils and transfers elsewhere (1e-13; FP32 2e-5)."""
import numpy as np
import pytest
import torch

from gpu_common import dev, handle_for, host, oracle_levels, problem, rel_inf
from oracle import ns as N
from oracle import tpmg as O
from synthetic import make_ns_problem

pytestmark = pytest.mark.gpu


def shifted(t):
    """The same values in a buffer one value off alignment."""
    buf = torch.empty(t.numel() + 1, dtype=t.dtype, device="cuda")
    out = buf[1:].view(t.shape)
    out.copy_(t)
    return out


# 5 x 4 and 7 x 6: odd longitudes take the column walk
STENCIL = [(4, 2, 1), (4, 2, 3), (5, 4, 3), (6, 4, 9), (34, 6, 13), (130, 66, 33), (256, 130, 9)]


@pytest.mark.parametrize("shape", STENCIL, ids=lambda s: "x".join(map(str, s)))
def test_stencil(shape):
    P = problem(*shape, sigma=0.2, seed=sum(shape))
    lev, _ = oracle_levels(P, levels=1)
    H = handle_for(P, levels=1)
    rng = np.random.default_rng(sum(shape))
    x, b = rng.standard_normal(lev[0].shape), rng.standard_normal(lev[0].shape)
    want = O.apply(lev[0], x)
    got = H.level_apply(0, dev(x))
    assert rel_inf(host(got), want) <= 1e-13
    assert torch.equal(got, H.level_apply(0, shifted(dev(x))))  # the column walk, bit for bit
    assert rel_inf(host(H.level_residual(0, dev(b), dev(x))), O.residual(lev[0], b, x)) <= 1e-13


@pytest.mark.parametrize("shape", [(4, 2, 3), (34, 6, 13), (66, 34, 9)],
                         ids=lambda s: "x".join(map(str, s)))
def test_directed_stencil(shape):
    from paper_2307_04528_gb300.solver import NSHandle
    names = ("h", "tx", "ty", "tz", "txr", "tyr", "tzr")
    P = make_ns_problem(*shape, 0.2, 31, pe=0.3)
    p = O.MGParams(levels=1)
    levs = N.build_hierarchy(*(P[k] for k in names), p)
    H = NSHandle(*(dev(P[k]) for k in names), levels=1)
    x = np.random.default_rng(3).standard_normal(P["h"].shape)
    for tr, lev in ((False, levs[0]), (True, N.transposed(levs)[0])):
        got = H.apply(dev(x), transpose=tr)
        assert rel_inf(host(got), N.apply(lev, x)) <= 1e-13
        assert torch.equal(got, H.apply(shifted(dev(x)), transpose=tr))


# 8: two quads to a row, rows ending inside a warp; 20 and 132: five and 33
# quads; 6: no whole quad
@pytest.mark.parametrize("shape", [(8, 4, 3), (20, 10, 7), (132, 34, 5), (6, 6, 4), (128, 64, 21)],
                         ids=lambda s: "x".join(map(str, s)))
def test_prolongation(shape):
    P = problem(*shape, sigma=0.2, seed=sum(shape))
    lev, _ = oracle_levels(P, levels=2)
    H = handle_for(P, levels=2)
    rng = np.random.default_rng(sum(shape))
    e, u = rng.standard_normal(lev[1].shape), rng.standard_normal(lev[0].shape)
    for prec, l0, dt, tol in ((0, lev[0], np.float64, 1e-13),
                              (1, O.float_levels(lev)[0], np.float32, 2e-5)):
        ee, uu = e.astype(dt), u.astype(dt)
        ref = uu.copy()
        O.prolong_add(l0, ee, ref)
        te, tu = (dev(a, torch.float64 if prec == 0 else torch.float32) for a in (ee, uu))
        assert rel_inf(host(H.level_prolong_add(0, te, tu.clone(), prec=prec)), ref) <= tol
        assert rel_inf(host(H.level_prolong_add(0, te, shifted(tu), prec=prec)), ref) <= tol
