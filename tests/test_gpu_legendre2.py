"""The two-degree Legendre kernels of FP64 plans (legendre2.cu) against the
one-degree recurrence with FP64 sums (fp64_contraction) on the same plan
sizes: every block size of the adjoint, ring counts off a multiple of 32,
fewer orders than degrees, both parities of lmax - m at the last step.

Tolerance: a sum of n float-pair products carries at most n 2^-47 of its
terms' size; both plans share the NUFFT kernel, whose own rounding is below
1e-12.
"""
import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu


def _pts(n, seed):
    p = W.points_uniform(n, seed)
    p[:4, 0] = [0.0, np.pi, np.pi / 2, 1e-9]  # both poles, the equator, next to a pole
    return p


@pytest.mark.parametrize("lmax,mmax", [(0, 0), (1, 1), (2, 0), (3, 2), (31, 31), (63, 63), (64, 64), (130, 7),
                                       (255, 254), (517, 301), (1023, 1023), (1700, 1700)])
def test_two_degree_against_one_degree(lmax, mmax):
    import torch

    import paper_2406_14542_gb300 as nu

    n = 4000
    pts = torch.from_numpy(_pts(n, lmax)).cuda()
    a = torch.from_numpy(W.alm_gaussian(lmax, seed=lmax + 1, mmax=mmax)).cuda()
    y = torch.from_numpy(np.random.default_rng(lmax).standard_normal(n)).cuda()
    two = nu.Plan(lmax, pts, eps=1e-12, precision="fp64", mmax=mmax)
    one = nu.Plan(lmax, pts, eps=1e-12, precision="fp64", mmax=mmax, fp64_contraction=True)
    tol = max(1e-12, lmax * 2.0**-47)
    for u, v in ((two.synth(a), one.synth(a)), (two.adjoint(y), one.adjoint(y)),
                 (two.adjoint_grad(y), one.adjoint_grad(y))):
        assert torch.isfinite(torch.view_as_real(u) if u.is_complex() else u).all()
        assert ((u - v).norm() / v.norm()).item() <= tol
    two.close()
    one.close()


@pytest.mark.parametrize("lmax,mmax", [(0, 0), (1, 1), (2, 0), (3, 2), (31, 31), (63, 63), (130, 7), (255, 254),
                                       (256, 256), (517, 301), (1023, 1023)])
def test_two_degree_table_against_recurrence(lmax, mmax):
    """Mixed plans: the two-degree table (both block kinds) against the
    per-call recurrence.  FP32 sums of up to lmax terms differ by at most
    lmax 2^-23 of their terms, and by a few 2^-24 from the stages they share."""
    import torch

    import paper_2406_14542_gb300 as nu

    n = 4000
    pts = torch.from_numpy(_pts(n, lmax)).cuda()
    a = torch.from_numpy(W.alm_gaussian(lmax, seed=lmax + 1, mmax=mmax, dtype=np.complex64)).cuda()
    y = torch.from_numpy(np.random.default_rng(lmax).standard_normal(n).astype(np.float32)).cuda()
    tab = nu.Plan(lmax, pts, eps=1e-5, precision="mixed", mmax=mmax)
    rec = nu.Plan(lmax, pts, eps=1e-5, precision="mixed", mmax=mmax, legendre_table=-1)
    tol = max(2e-6, lmax * 2.0**-23)
    for u, v in ((tab.synth(a), rec.synth(a)), (tab.adjoint(y), rec.adjoint(y)),
                 (tab.adjoint_grad(y), rec.adjoint_grad(y))):
        assert torch.isfinite(torch.view_as_real(u) if u.is_complex() else u).all()
        assert ((u - v).norm() / v.norm()).item() <= tol
    tab.close()
    rec.close()
