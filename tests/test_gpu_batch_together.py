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
    """A batch whose FP32 solves all run on their own times its work lists on the
    FP64 sweeps in its first FP64 solve: at least eight widths and grids, four
    launches each; and only there."""
    from paper_2307_04528_gb300.solver import MGBatch
    p = problem(256, 128, 65, sigma=0.1, seed=70)
    B = MGBatch([tuple(dev(p[k]) for k in ("tx", "ty", "tz", "h"))], mixed=1)
    b = dev(p["b"])
    count = []
    for _ in range(3):
        n0 = launches()
        x, info = B.solve([b], tol=1e-9, mixed=0)
        count.append(launches() - n0)
        assert info[0]["status"] == 0 and info[0]["rel_res"] <= 1e-9
    assert count[0] >= count[1] + 32 and count[1] == count[2]
