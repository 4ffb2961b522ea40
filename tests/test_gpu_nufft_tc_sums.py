"""Tensor-core spreading (nufft_tc.cu) of many points whose products have one
sign: positions hit again and again with one value (a hit count at pixel
centres), points crowded in a few bins, points on one colatitude.  A block then
sums up to eight subproblems of one bin before it writes the tile.

Tolerance: as for other inputs (test_gpu_nufft_tc.py): the digit products drop
terms below 2^-48 of the operands' scales, float pairs in the other stages
~2^-47 per operation, the deconvolution's factors at the band edge on both:
1e-12 against FP64 instructions.
"""
import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu


def _points(kind, n):
    rng = np.random.default_rng(2)
    if kind == "positions":
        return W.points_uniform(6, 5)[rng.integers(0, 6, n)]
    if kind == "colatitude":
        return np.stack([np.full(n, 1.1), 2.0 + 0.02 * rng.random(n)], axis=1)
    return np.stack([1.0 + 0.02 * rng.random(n), 2.0 + 0.02 * rng.random(n)], axis=1)


@pytest.mark.parametrize("eps", [1e-10, 1e-11, 1e-12])  # w = 14, 16, 17
@pytest.mark.parametrize("kind,n", [("positions", 1536), ("positions", 4000000), ("crowd", 1500000),
                                    ("colatitude", 1500000)])
def test_constant_map_on_crowded_points(kind, n, eps):
    import torch

    import paper_2406_14542_gb300 as nu

    pts = torch.from_numpy(np.ascontiguousarray(_points(kind, n))).cuda()
    y = torch.ones(n, dtype=torch.float64, device="cuda")
    plan = nu.Plan(95, pts, eps=eps)
    ref = nu.Plan(95, pts, eps=eps, fp64_contraction=True, fft_kernels=-1)
    u, v = plan.adjoint(y), ref.adjoint(y)
    assert ((u - v).norm() / v.norm()).item() <= 1e-12
    plan.close()
    ref.close()
