"""Batch members large enough to be solved on their own beside members in lock
step (the line is at 2^21 cells): the same bits as their single-system solves,
and their statuses next to the others' (a non-finite and a zero right-hand
side, an iteration limit)."""
import pytest
import torch

from gpu_common import dev, problem

pytestmark = pytest.mark.gpu

SHAPES = [(256, 128, 64), (64, 32, 16), (256, 128, 65), (256, 128, 63)]


def batch(**params):
    from paper_2307_04528_gb300.solver import MGBatch
    probs = [problem(*s, sigma=0.1, seed=40 + i) for i, s in enumerate(SHAPES)]
    B = MGBatch([tuple(dev(P[k]) for k in ("tx", "ty", "tz", "h")) for P in probs], mixed=1,
                **params)
    return B, [dev(P["b"]) for P in probs]


def test_same_as_single():
    B, bs = batch()
    xs, infos = B.solve(bs, tol=1e-9)
    for i in (0, 2):
        x, info = B.handle(i).solve_mixed(bs[i], tol=1e-9)
        assert torch.equal(x, xs[i])
        for k in ("status", "iterations", "inner_iterations", "rel_res"):
            assert info[k] == infos[i][k], k
    assert all(v["status"] == 0 and v["rel_res"] <= 1e-9 for v in infos)


@pytest.mark.parametrize("which", [0, 3])
def test_statuses(which):
    from paper_2307_04528_gb300 import _lib as L
    B, bs = batch()
    bs[which][0, 0, 0] = float("nan")
    bs[2].zero_()
    xs, infos = B.solve(bs, tol=1e-9, raise_on_error=False)
    want = [0] * len(SHAPES)
    want[which] = L.MG_ERR_NONFINITE
    assert [v["status"] for v in infos] == want
    assert infos[which]["iterations"] == 0 and not torch.any(xs[which])
    assert infos[2]["iterations"] == 0 and infos[2]["rel_res"] == 0 and not torch.any(xs[2])


def test_limit():
    from paper_2307_04528_gb300 import _lib as L
    B, bs = batch(maxit=1, inner_maxit=2)
    _, infos = B.solve(bs, tol=1e-12, raise_on_error=False)
    for v in infos:
        assert v["status"] == L.MG_ERR_NOT_CONVERGED
        assert v["iterations"] == 1 and v["inner_iterations"] == 2
