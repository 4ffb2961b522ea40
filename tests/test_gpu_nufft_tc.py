"""Tensor-core interpolation and spreading of FP64 plans (nufft_tc.cu) against
the FP64-instruction kernels (fp64_contraction) on the same points: bins at
the grid's edge and wrapping halos, subproblems of every fill (a last group of
one point, many subproblems of one bin, empty bins between runs), repeated
points, both kernel-width parities up to the widest tile, deterministic mode.

Tolerance: both use the same kernel values; the digit products drop terms
below 2^-48 of the operands' scales, float pairs in the other stages ~2^-47
per operation, against sums of up to a few hundred terms: 1e-12.
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
    elif kind == "same":  # one point many times
        p = np.tile([[1.2345, 3.21]], (n, 1))
    else:  # around phi = 0 = 2 pi and over the south pole (theta beyond pi)
        p = np.stack([np.pi + 0.3 * (rng.random(n) - 0.5), 0.2 * (rng.random(n) - 0.5)], axis=1)
    return np.ascontiguousarray(p)


@pytest.mark.parametrize("eps", [1e-8, 1e-10, 1e-11, 1e-12])  # w = 12, 14, 15, 17
@pytest.mark.parametrize("kind,lmax,n", [("sphere", 40, 5000), ("sphere", 200, 30001), ("sphere", 511, 200000),
                                         ("cluster", 95, 5001), ("same", 63, 700), ("wrap", 127, 4097)])
def test_tensor_core_nufft_against_fp64(kind, lmax, n, eps):
    import torch

    import paper_2406_14542_gb300 as nu

    pts = torch.from_numpy(_points(kind, n, lmax)).cuda()
    a = torch.from_numpy(W.alm_gaussian(lmax, seed=lmax)).cuda()
    y = torch.from_numpy(np.random.default_rng(n).standard_normal(n)).cuda()
    tc = nu.Plan(lmax, pts, eps=eps, precision="fp64")
    det = nu.Plan(lmax, pts, eps=eps, precision="fp64", deterministic=True)
    ref = nu.Plan(lmax, pts, eps=eps, precision="fp64", fp64_contraction=True, fft_kernels=-1)
    for u, v in ((tc.synth(a), ref.synth(a)), (tc.adjoint(y), ref.adjoint(y)), (det.adjoint(y), ref.adjoint(y))):
        assert ((u - v).norm() / v.norm()).item() <= 1e-12
    assert torch.equal(det.adjoint(y), det.adjoint(y))
    for p in (tc, det, ref):
        p.close()


def test_tensor_core_nufft_nan_and_zero():
    """A NaN among the values reaches the coefficients, a NaN coefficient the
    map; zero inputs give zeros, also after a call that left the grid full."""
    import torch

    import paper_2406_14542_gb300 as nu

    n, lmax = 6000, 60
    pts = torch.from_numpy(W.points_uniform(n, 3)).cuda()
    a = torch.from_numpy(W.alm_gaussian(lmax, seed=1)).cuda()
    plan = nu.Plan(lmax, pts, eps=1e-10, precision="fp64")
    f = plan.synth(a)
    assert plan.adjoint(torch.zeros_like(f)).abs().max().item() == 0.0
    assert plan.synth(torch.zeros_like(a)).abs().max().item() == 0.0
    bad = f.clone()
    bad[1234] = float("nan")
    assert torch.isnan(plan.adjoint(bad).real).any()
    b = a.clone()
    b[100] = float("nan")
    assert torch.isnan(plan.synth(b)).any()
    assert ((plan.synth(a) - f).norm() / f.norm()).item() == 0.0
    plan.close()
