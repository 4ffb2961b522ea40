"""Tensor-core spreading (nufft_tc.cu) of values from the whole double range
next to ordinary ones in the same bins: what lies below 2^-74 of a block's
largest value, down to the smallest normal number and subnormals, counts as
zero.

Tolerance: the same operands as with zeros in those places, so the same bits
in deterministic mode; the atomics' order otherwise (1e-13).
"""
import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu

SMALL = [2.0**-1022, -(2.0**-1022), 1e-307, 1e-306, -1e-305, 1e-303, 1e-300, 1e-310, 5e-324]


def _cuda(x):
    import torch

    return torch.from_numpy(np.ascontiguousarray(x)).cuda()


@pytest.mark.parametrize("deterministic", [False, True])
@pytest.mark.parametrize("top", [4.0, 1e3, 1e12, 1e30])
def test_small_values_next_to_ordinary_ones(top, deterministic):
    import torch

    import paper_2406_14542_gb300 as nu

    lmax, n = 200, 60000
    rng = np.random.default_rng(int(np.log10(top)))
    pts = _cuda(W.points_uniform(n, 1))
    y = 2.0 + (top - 2.0) * rng.random(n)
    small = rng.random(n) < 0.3
    zeros = np.where(small, 0.0, y)
    y[small] = np.resize(SMALL, int(small.sum()))
    plan = nu.Plan(lmax, pts, eps=1e-10, deterministic=deterministic)
    for f in (plan.adjoint, plan.adjoint_grad):
        u, v = f(_cuda(y)), f(_cuda(zeros))
        if deterministic:
            assert torch.equal(u, v)
        assert ((u - v).norm() / v.norm()).item() <= 1e-13
    plan.close()
