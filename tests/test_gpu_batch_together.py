"""Batch members of 2^21 to 7 2^20 cells take part in the lock step where enough of
them share it: fewer launches than one solve after the other, and the solutions of
the single-system solves (residuals below 1e-9, solutions to 1e-7: the condition of
these systems times that)."""
import pytest
import torch

from gpu_common import dev, host, problem, rel_2

pytestmark = pytest.mark.gpu


def launches():
    from paper_2307_04528_gb300 import load
    return load().mg_launch_count()


def test_many_of_middle_size():
    from paper_2307_04528_gb300.solver import MGBatch
    P = [problem(256, 128, 65, sigma=0.1, seed=70 + i) for i in range(2)]
    probs = [P[i % 2] for i in range(6)]
    B = MGBatch([tuple(dev(p[k]) for k in ("tx", "ty", "tz", "h")) for p in probs], mixed=1)
    bs = [dev(p["b"]) for p in probs]
    n0 = launches()
    xs, infos = B.solve(bs, tol=1e-9)
    batch = launches() - n0
    n0 = launches()
    alone = [B.handle(i).solve_mixed(bs[i], tol=1e-9)[0] for i in range(2)]
    single = (launches() - n0) / 2
    assert batch < 3 * single  # of six
    for i, (x, info) in enumerate(zip(xs, infos)):
        assert info["status"] == 0 and info["rel_res"] <= 1e-9
        assert rel_2(host(x), host(alone[i % 2])) <= 1e-7


def test_work_lists_tuned_without_fp32_members():
    """A batch whose FP32 solves all run on their own still times its work lists
    (the FP64 ones) at setup: at least eight widths and grids, four launches each."""
    from paper_2307_04528_gb300.solver import MGBatch, MGHandle
    p = problem(256, 128, 65, sigma=0.1, seed=70)
    fields = tuple(dev(p[k]) for k in ("tx", "ty", "tz", "h"))
    n0 = launches()
    MGHandle(*fields, mixed=1)
    handle = launches() - n0
    n0 = launches()
    B = MGBatch([fields], mixed=1)
    assert launches() - n0 >= handle + 32
    b = dev(p["b"])
    x, info = B.solve([b], tol=1e-9, mixed=0)
    assert info[0]["status"] == 0 and info[0]["rel_res"] <= 1e-9
