"""V-cycles and operator applications by direct launches, whose kernels are placed
while the one before them drains, against the same calls captured in a graph,
whose kernels wait for the whole of it: the same bits, over many passes in which
every buffer changes between passes."""
import pytest
import torch

from gpu_common import dev, handle_for, problem
from synthetic import make_ns_problem

pytestmark = pytest.mark.gpu

NAMES = ("h", "tx", "ty", "tz", "txr", "tyr", "tzr")


def compare(call, inputs):
    static = inputs[0].clone()
    side = torch.cuda.Stream()
    side.wait_stream(torch.cuda.current_stream())
    with torch.cuda.stream(side):
        call(static)
    torch.cuda.current_stream().wait_stream(side)
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        out = call(static)
    want = []
    for t in inputs:
        static.copy_(t)
        g.replay()
        want.append(out.clone())
    torch.cuda.synchronize()
    for _ in range(10):
        got = [call(t) for t in inputs]  # back to back
        for a, b in zip(got, want):
            assert torch.equal(a, b)


@pytest.mark.parametrize("prec", [0, 1])
@pytest.mark.parametrize("shape", [(64, 32, 16), (88, 50, 13), (256, 128, 30)],
                         ids=lambda s: "x".join(map(str, s)))
def test_symmetric(shape, prec):
    H = handle_for(problem(*shape, sigma=0.2, seed=5))
    dt = torch.float64 if prec == 0 else torch.float32
    gen = torch.Generator(device="cuda").manual_seed(1)
    rs = [torch.randn(shape[::-1], generator=gen, device="cuda", dtype=dt) for _ in range(4)]
    compare(lambda t: H.vcycle(t, prec=prec), rs)
    if prec == 0:
        compare(lambda t: H.apply(H.vcycle(t)), rs)


@pytest.mark.parametrize("prec", [0, 1])
def test_directed(prec):
    from paper_2307_04528_gb300.solver import NSHandle
    P = make_ns_problem(128, 66, 20, 0.2, 9, pe=0.3)
    H = NSHandle(*(dev(P[k]) for k in NAMES), mixed=1)
    dt = torch.float64 if prec == 0 else torch.float32
    gen = torch.Generator(device="cuda").manual_seed(2)
    rs = [torch.randn((20, 66, 128), generator=gen, device="cuda", dtype=dt) for _ in range(4)]
    for tr in (False, True):
        compare(lambda t: H.vcycle(t, transpose=tr, prec=prec), rs)
