"""Responses and gradients with the tile shape chosen by size (128 x 64, 256 x 128, 256 x 256)
against pair tiles of 256 x 256, on both sides of each change of shape: the same products in
the same order, and a layer's records the same, so the same bits, statistics included."""
import ctypes

import pytest
import torch

import paper_2107_02737_gb300.sp2 as sp2
from tests.test_gpu_tile_shapes import random_system

pytestmark = pytest.mark.gpu


def adjoint(H, G, cta_group, fwd=None, stride=0):
    """sp2_adjoint with the tile shape as given (the Python entry point leaves it to the library)."""
    n = H.shape[0]
    o = sp2.make_opts("fp16", cta_group=cta_group, checkpoint_stride=stride)
    D, dH = (torch.empty((n, n), dtype=torch.float32, device="cuda") for _ in range(2))
    st = sp2._new_stats()
    s = sp2.load().sp2_adjoint(ctypes.c_void_p(H.data_ptr()), ctypes.c_void_p(G.data_ptr()), n, float(n // 2), 1e-6,
                               ctypes.byref(fwd.raw) if fwd is not None else None, ctypes.c_void_p(D.data_ptr()),
                               ctypes.c_void_p(dH.data_ptr()), ctypes.byref(st), ctypes.byref(o), None, 0,
                               ctypes.c_void_p(torch.cuda.current_stream().cuda_stream))
    assert s == sp2.OK
    return D, dH, sp2._result(s, st)


@pytest.mark.parametrize("n,shape", [(65, 1), (300, 1), (1408, 1), (1409, 2), (2048, 2)])
@pytest.mark.parametrize("stride", [0, 4])
def test_adjoint(n, shape, stride):
    H, G = random_system(n, n), random_system(n, n + 1)
    D0, g0, r0 = adjoint(H, G, 0, stride=stride)
    D1, g1, r1 = adjoint(H, G, 2, stride=stride)
    assert r0.cta_group == shape and r1.cta_group == 2
    assert torch.equal(D0, D1) and torch.equal(g0, g1)
    assert r0.choices == r1.choices and r0.trace == r1.trace and r0.trace_sq == r1.trace_sq
    # and with the layers of an earlier forward run replayed
    _, fwd = sp2.density(H, n // 2)
    _, g2, r2 = adjoint(H, G, 0, fwd, stride)
    _, g3, r3 = adjoint(H, G, 2, fwd, stride)
    assert torch.equal(g2, g3) and r2.trace == r3.trace


@pytest.mark.parametrize("n,shape", [(65, 1), (1024, 1), (1025, 2), (1408, 2), (1409, 2)])
def test_response(n, shape):
    H, M = random_system(n, n), random_system(n, n + 1)
    D0, R0, r0 = sp2.response(H, M, n // 2)
    D1, R1, r1 = sp2.response(H, M, n // 2, cta_group=2)
    assert r0.cta_group == shape and r1.cta_group == 2
    assert torch.equal(D0, D1) and torch.equal(R0, R1)
    assert r0.trace == r1.trace and r0.trace_sq == r1.trace_sq
