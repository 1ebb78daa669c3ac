"""The conjugate-gradient iterations as a loop on the device against the same
iterations driven by the host (which run while profiling is on): the same
kernels in the same order, so histories and solutions agree bit for bit, and
the calls end alike: converged, at the iteration limit (also past the 256
norms that one launch of the loop records), and from an x the loop refuses."""
import pytest
import torch

from gpu_common import dev, handle_for, problem

pytestmark = pytest.mark.gpu


def both(shape, call, **params):
    P = problem(*shape, sigma=0.2, seed=11)
    H = handle_for(P, **params)
    out = []
    for host_loop in (False, True):
        H.profile(host_loop)
        b = dev(P["b"])
        x, info = call(H, b)
        out.append((x.clone(), info))
    (x, a), (y, c) = out
    assert torch.equal(x, y)
    assert a["status"] == c["status"]
    assert a["iterations"] == c["iterations"] and list(a["history"]) == list(c["history"])
    return a


@pytest.mark.parametrize("name", ["solve", "solve_mixed"])
@pytest.mark.parametrize("shape", [(6, 4, 3), (18, 10, 5), (64, 32, 16)],
                         ids=lambda s: "x".join(map(str, s)))
def test_converged(shape, name):
    info = both(shape, lambda H, b: getattr(H, name)(b, tol=1e-9))
    assert info["iterations"] >= 1


@pytest.mark.parametrize("offset", [0, 1])
def test_single_precision_x_of_any_alignment(offset):
    def call(H, b):
        buf = torch.zeros(b.numel() + 1, dtype=torch.float32, device="cuda")
        return H.solve_single(b.float(), x=buf[offset:offset + b.numel()].view(b.shape), tol=1e-4,
                              raise_on_error=False)  # FP32 ends at its floor, restarting
    both((20, 10, 9), call)


@pytest.mark.parametrize("maxit", [1, 255, 256, 257, 600])
def test_iteration_limit(maxit):
    # one level, one weak sweep: far from the tolerance at every limit
    info = both((64, 32, 3), lambda H, b: H.solve(b, tol=1e-300, history_cap=1024,
                                                 raise_on_error=False),
                levels=1, coarse_iters=1, maxit=maxit)
    assert info["iterations"] == maxit


# FP32 adds two directions to x every other iteration: both parities of the
# last one, of one launch and of several
@pytest.mark.parametrize("maxit", [1, 2, 3, 256, 257, 513])
@pytest.mark.parametrize("shape", [(64, 32, 3), (65, 34, 3)], ids=["quads", "values"])
def test_single_precision_limit(shape, maxit):
    info = both(shape, lambda H, b: H.solve_single(b.float(), tol=1e-30, raise_on_error=False),
                levels=1, coarse_iters=1, maxit=maxit)
    assert info["iterations"] == maxit
