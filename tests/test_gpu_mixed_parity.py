"""The mixed adjoint's even and odd degrees (l - m) each against an FP64 plan
with the same points: in ring blocks away from the equator the even ones follow
from the odd degrees' table (legtab.cu), with factors 1 / cos(theta) of up to 4.
Maps over the sphere, in the polar caps and in the bands where that factor is
largest.

Tolerance: half of the plan's eps of 1e-5.  The spreading kernel takes 1e-6 of it,
FP32 rounding in sums of up to lmax terms of random sign a few sqrt(lmax) 2^-24.
"""
import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("lmax", [63, 255, 1023, 2047])
def test_even_and_odd_degrees_of_the_mixed_adjoint(lmax):
    import torch

    import paper_2406_14542_gb300 as nu

    n = min(4 * (lmax + 1) ** 2, 1500000)
    p = W.points_uniform(n, lmax)
    pts = torch.from_numpy(p).cuda()
    x = np.abs(np.cos(p[:, 0]))
    rng = np.random.default_rng(lmax)
    even = torch.from_numpy(np.concatenate([np.arange(lmax + 1 - m) % 2 == 0 for m in range(lmax + 1)])).cuda()
    mixed = nu.Plan(lmax, pts, eps=1e-5, precision="mixed")
    exact = nu.Plan(lmax, pts, eps=1e-10)
    for where in (x >= 0, x > 0.98, (x > 0.25) & (x < 0.35)):
        y = torch.from_numpy(np.where(where, rng.standard_normal(n), 0.0).astype(np.float32)).cuda()
        u, v = mixed.adjoint(y).to(torch.complex128), exact.adjoint(y.double())
        for s in (even, ~even):
            assert ((u - v)[s].norm() / v[s].norm()).item() <= 5e-6
    mixed.close()
    exact.close()
