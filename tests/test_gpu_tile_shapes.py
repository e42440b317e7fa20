"""The tensor-core tile shapes chosen by size (128 x 64, 256 x 128, 256 x 256) compute each
element from the same products in the same order, and a layer's
the same bit for bit with every shape: sizes on both sides of each change of shape and
ragged ones."""
import pytest
import torch

import paper_2107_02737_gb300.sp2 as sp2

pytestmark = pytest.mark.gpu


def random_system(n, seed):
    g = torch.Generator(device="cuda").manual_seed(seed)
    a = torch.randn(n, n, generator=g, device="cuda", dtype=torch.float64)
    q, _ = torch.linalg.qr(a)
    lam = torch.rand(n, generator=g, device="cuda", dtype=torch.float64) * 0.95 + 0.05
    lam[: n // 2] *= -1.0
    H = (q * lam) @ q.T
    return (H + H.T) / 2


@pytest.mark.parametrize("n", [2, 65, 257, 1408, 1409, 2048, 2049, 2816])
@pytest.mark.parametrize("precision", ["fp16", "bf16"])
def test_density_is_the_same_with_every_tile_shape(n, precision):
    H = random_system(n, n)
    D0, r0 = sp2.density(H, n // 2, precision=precision)
    D, r = sp2.density(H, n // 2, precision=precision, cta_group=2)
    assert torch.equal(D, D0)
    assert r.choices == r0.choices and r.trace == r0.trace and r.trace_sq == r0.trace_sq


@pytest.mark.parametrize("n", [300, 1100, 1700])
def test_response_and_adjoint_are_the_same_with_every_tile_shape(n):
    H, M = random_system(n, n), random_system(n, n + 1)
    D, res = sp2.density(H, n // 2)
    for gap in (None, (-0.04, 0.04)):
        D0, R0, _ = sp2.response(H, M, n // 2, gap=gap)
        D1, R1, _ = sp2.response(H, M, n // 2, gap=gap, cta_group=2)
        assert torch.equal(D0, D1) and torch.equal(R0, R1)
    _, g0, _ = sp2.adjoint(H, M, n // 2, fwd=res)
    _, g1, _ = sp2.adjoint(H, M, n // 2, fwd=res, checkpoint_stride=4)
    assert torch.equal(g0, g1)
