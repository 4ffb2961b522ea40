"""Tensor-core spreading and interpolation (nufft_tc.cu) with a kernel error
near rounding: maps whose values span decades inside every bin (bright pixels
over a faint field), which share one scale per block.

Tolerance: that of float pairs in every stage, ~2^-47 per operation raised by
the deconvolution's factors at the band edge: 1e-13 against FP64 instructions
(the float-pair kernels have 4e-14 on these maps).
"""
import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("eps", [1e-11, 1e-12])  # w = 16, 17
@pytest.mark.parametrize("decades", [0, 3, 6])
def test_maps_with_a_wide_range(decades, eps):
    import torch

    import paper_2406_14542_gb300 as nu

    lmax, n = 95, 30000
    rng = np.random.default_rng(decades)
    pts = torch.from_numpy(W.points_uniform(n, 3)).cuda()
    y = torch.from_numpy(rng.standard_normal(n) * 10.0 ** (-decades * rng.random(n) ** 0.1)).cuda()
    a = torch.from_numpy(W.alm_gaussian(lmax, seed=4)).cuda()
    plan = nu.Plan(lmax, pts, eps=eps)
    ref = nu.Plan(lmax, pts, eps=eps, fp64_contraction=True, fft_kernels=-1)
    for u, v in ((plan.adjoint(y), ref.adjoint(y)), (plan.synth(a), ref.synth(a))):
        assert ((u - v).norm() / v.norm()).item() <= 1e-13
    plan.close()
    ref.close()
