"""FP32 spreading by one warp per subproblem (scattered points, w = 6..8,
at least 2048 subproblems) against the deterministic mode's kernel, which adds
the same kernel values in a fixed order: bins at the grid's edge and wrapping
halos, subproblems of one point and of all sizes, many of one bin, repeated
points; a batch of uneven members against the members' own plans.

Tolerance: both round products and sums of the same FP32 kernel values; up to
6e5 values of random sign meet in one cell, in subproblems of 256 whose sums
are added in turn: (sqrt(256) + sqrt(2400)) 2^-24 < 4e-6 of the result, and
FP32 rounding of a few 1e-7 in the stages after it: 1e-5.
"""
import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu


def _points(kind, n, seed):
    rng = np.random.default_rng(seed)
    if kind == "sphere":
        p = W.points_uniform(n, seed)
        p[:3, 0] = [0.0, np.pi, np.pi / 2]
    elif kind == "cluster":  # nearly all points in one bin
        p = np.stack([1.0 + 1e-3 * rng.random(n), 2.0 + 1e-3 * rng.random(n)], axis=1)
        p[: n // 16] = W.points_uniform(n // 16, seed + 1)
    else:  # around phi = 0 = 2 pi and over the south pole (theta beyond pi)
        p = np.stack([np.pi + 0.3 * (rng.random(n) - 0.5), 0.2 * (rng.random(n) - 0.5)], axis=1)
    return np.ascontiguousarray(p)


@pytest.mark.parametrize("eps", [1e-4, 1e-5, 1e-6])  # w = 6, 7, 8
@pytest.mark.parametrize("kind,lmax,n", [("sphere", 700, 400001), ("sphere", 1023, 2000003), ("cluster", 95, 600001),
                                         ("wrap", 255, 600007)])
def test_warp_spreading_against_ordered(kind, lmax, n, eps):
    import torch

    import paper_2406_14542_gb300 as nu

    pts = torch.from_numpy(_points(kind, n, lmax)).cuda()
    y = torch.from_numpy(np.random.default_rng(n).standard_normal(n).astype(np.float32)).cuda()
    plan = nu.Plan(lmax, pts, eps=eps, precision="mixed")
    det = nu.Plan(lmax, pts, eps=eps, precision="mixed", deterministic=True)
    assert 6 <= plan.info()["w"] <= 8
    u, v = plan.adjoint(y), det.adjoint(y)
    assert ((u - v).norm() / v.norm()).item() <= 1e-5
    assert plan.adjoint(torch.zeros_like(y)).abs().max().item() == 0.0
    plan.close()
    det.close()


def test_warp_spreading_batch():
    import torch

    import paper_2406_14542_gb300 as nu

    ls = [300, 31, 511, 64]
    pts = [torch.from_numpy(_points("sphere", n, n)).cuda() for n in (180001, 33, 300000, 5000)]
    ys = [torch.from_numpy(np.random.default_rng(i).standard_normal(len(p)).astype(np.float32)).cuda()
          for i, p in enumerate(pts)]
    bp = nu.BatchPlan(ls, pts, eps=1e-5)
    out = bp.adjoint(ys)
    for l, p, y, u in zip(ls, pts, ys, out):
        det = nu.Plan(l, p, eps=1e-5, precision="mixed", deterministic=True)
        v = det.adjoint(y)
        assert ((u - v).norm() / v.norm()).item() <= 1e-5
        det.close()
    bp.close()
