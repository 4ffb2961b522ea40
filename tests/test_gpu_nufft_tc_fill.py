"""The rule that takes a point set to the tensor-core interpolation and
spreading (nufft_tc.cu): points per bin on either side of each kernel width's
line, in one plan whose points are set anew, so that the stored kernel values
change their format each time.  Synthesis, adjoint and gradient against FP64
instructions.

Tolerance: that of test_gpu_nufft_tc.py (1e-12); gradients carry the factor of
the derivative, up to lmax, on the same rounding: 1e-12 of their norm.
"""
import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("eps", [1e-8, 1e-9, 1e-10, 1e-11])  # w = 12, 13, 14, 16
def test_points_per_bin_on_either_side_of_the_line(eps):
    import torch

    import paper_2406_14542_gb300 as nu

    lmax = 639
    bins = 7100  # of 16 x 16 cells on the half of the fine grid that the sphere covers
    a = torch.from_numpy(W.alm_gaussian(lmax, seed=4)).cuda()
    plan = ref = None
    for k, fill in enumerate((45, 14, 36, 18, 24, 12)):
        n = fill * bins
        pts = torch.from_numpy(W.points_uniform(n, k)).cuda()
        y = torch.from_numpy(np.random.default_rng(k).standard_normal(n)).cuda()
        if plan is None:
            plan = nu.Plan(lmax, pts, eps=eps)
            ref = nu.Plan(lmax, pts, eps=eps, fp64_contraction=True, fft_kernels=-1)
        else:
            plan.setpts(pts)
            ref.setpts(pts)
        pairs = [(plan.synth(a), ref.synth(a)), (plan.adjoint(y), ref.adjoint(y))]
        pairs += list(zip(plan.synth_grad(a), ref.synth_grad(a)))
        for u, v in pairs:
            assert ((u - v).norm() / v.norm()).item() <= 1e-12
    plan.close()
    ref.close()
