"""The conjugate-gradient iterations run as a loop on the device where they can:
after an ordinary solve, and not while profiling, from an FP32 x off its 16-byte
boundary, or for another method (so that the comparisons of the loop with the
host-driven iterations compare two things)."""
import pytest
import torch

from gpu_common import dev, handle_for, problem

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shape", [(6, 4, 3), (64, 32, 16), (65, 34, 3)],
                         ids=lambda s: "x".join(map(str, s)))
def test_loop_runs(shape):
    P = problem(*shape, sigma=0.2, seed=11)
    b = dev(P["b"])
    H = handle_for(P)
    assert not H.device_loop(0) and not H.device_loop(1)
    H.profile(True)
    H.solve(b, tol=1e-9)
    H.solve_mixed(b, tol=1e-9)
    assert not H.device_loop(0) and not H.device_loop(1)
    H.profile(False)
    buf = torch.zeros(b.numel() + 1, dtype=torch.float32, device="cuda")
    H.solve_single(b.float(), x=buf[1:].view(b.shape), tol=1e-4, raise_on_error=False)
    assert not H.device_loop(1)
    H.solve(b, tol=1e-9)
    assert H.device_loop(0) and not H.device_loop(1)
    H.solve_mixed(b, tol=1e-9)
    assert H.device_loop(1)


def test_other_methods_have_none():
    P = problem(32, 16, 8, sigma=0.2, seed=3)
    H = handle_for(P, method=1)
    H.solve(dev(P["b"]), tol=1e-6, raise_on_error=False)
    assert not H.device_loop(0)
