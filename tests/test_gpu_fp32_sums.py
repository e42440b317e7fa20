"""Precision of the FP32 path's layer sums: ||X||_F^2 of one layer against the exactly
rounded sum.  A thread adds its elements as compensated FP32 pairs (some 2^-48 of its sum
each, and independent over the tens of thousands of threads, so below 2^-53 of the total);
everything above a thread is FP64, about twenty roundings of at most 2^-53 that add up like
a random walk: 5e-16.  Twice that is allowed; sums kept in FP32 pairs across a tile are
2e-15 off and more at these sizes."""
import math

import numpy as np
import pytest
import torch

import paper_2107_02737_gb300.sp2 as sp2

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [1700, 3000])
def test_sum_of_squares_is_summed_in_fp64(n):
    errs = []
    for seed in range(4):
        g = torch.Generator(device="cuda").manual_seed(1000 + seed)
        q, _ = torch.linalg.qr(torch.randn(n, n, generator=g, device="cuda", dtype=torch.float64))
        lam = torch.rand(n, generator=g, device="cuda", dtype=torch.float64)
        x = (q * lam) @ q.T
        X, res = sp2.apply_layers(((x + x.T) / 2).to(torch.float32), [0], precision="fp32")
        x = X.double().cpu().numpy()
        exact = math.fsum((x * x).ravel())
        errs.append(abs(res.trace_sq[1] - exact) / exact)
        assert abs(res.trace[1] - math.fsum(np.diag(x))) <= 1e-14 * n
    assert np.mean(errs) <= 1e-15, errs
