"""Sweeps and the coarsest-level solve on either side of the lines of their dispatch:
the column walks that large levels of many layers take (from zero and on a guess, in
both precisions), and cluster solves that fill a block's threads or miss by a row or a
column.  Against the CPU oracle at the tolerances of the sweeps elsewhere (FP64 1e-13,
twelve sweeps 1e-12; FP32 2e-5)."""
import numpy as np
import pytest
import torch

from gpu_common import dev, handle_for, host, oracle_levels, problem, rel_inf
from oracle import tpmg as O

pytestmark = pytest.mark.gpu


def both(shape):
    P = problem(*shape, sigma=0.2, seed=sum(shape))
    lev, p = oracle_levels(P, levels=1)
    H = handle_for(P, levels=1)
    rng = np.random.default_rng(sum(shape) + 3)
    b, u = rng.standard_normal(lev[0].shape), rng.standard_normal(lev[0].shape)
    for prec, ol in ((0, lev[0]), (1, O.float_levels(lev)[0])):
        dt = ol.h.dtype
        put = lambda a: dev(a, torch.float32 if prec else torch.float64)
        yield H, prec, ol, b.astype(dt), u.astype(dt), dt.type(p.omega), put


# 8192 columns and more: 76 layers fit no shape's waste rule, 81 no shape, 192 is the most
@pytest.mark.parametrize("shape", [(128, 64, 76), (128, 64, 81), (130, 64, 81), (128, 64, 192)],
                         ids=lambda s: "x".join(map(str, s)))
def test_walks(shape):
    for H, prec, ol, b, u, om, put in both(shape):
        zero, guess = np.zeros_like(b), u.copy()
        O.smooth(ol, b, zero, om)
        O.smooth(ol, b, guess, om)
        tol = 2e-5 if prec else 1e-13
        assert rel_inf(host(H.level_smooth(0, put(b), prec=prec)), zero) <= tol, prec
        assert rel_inf(host(H.level_smooth(0, put(b), put(u), prec=prec)), guess) <= tol, prec
        got, dot = H.level_smooth_dot(0, put(b), put(u), prec=prec)
        assert rel_inf(host(got), guess) <= tol, prec
        assert abs(dot - O.dot(b, guess)) <= tol * O.norm2(b) * O.norm2(guess)


# FP64 on either side of the line between segments and walk, by layers and by columns
@pytest.mark.parametrize("shape", [(32, 32, 4), (32, 32, 5), (64, 64, 16), (96, 80, 10),
                                   (64, 98, 50), (96, 80, 50), (128, 64, 70)],
                         ids=lambda s: "x".join(map(str, s)))
def test_fp64_segments_and_walk(shape):
    test_walks(shape)


# rows of eight blocks that just fit and just do not: 70 layers in 9 segments (FP32) and
# 18 (FP64), 100 layers in 9 and 17, one and two layers
@pytest.mark.parametrize("shape", [(8, 56, 70), (8, 58, 70), (14, 32, 70), (10, 16, 70),
                                   (10, 18, 70), (14, 8, 100), (16, 8, 100), (6, 4, 192),
                                   (64, 64, 1), (66, 64, 2), (4, 2, 1)],
                         ids=lambda s: "x".join(map(str, s)))
def test_coarsest_solve(shape):
    for H, prec, ol, b, _, om, put in both(shape):
        want = np.zeros_like(b)
        for _ in range(12):
            O.smooth(ol, b, want, om)
        tol = 2e-5 if prec else 1e-12
        assert rel_inf(host(H.level_relax(0, put(b), 12, prec=prec)), want) <= tol, prec
