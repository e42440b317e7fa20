"""FP32 CUDA-core layers at the edges of their tile sides (32, 64 and 128 by padded
size): one layer of each sign against the FP64 layer, and a batch that mixes the sides
against lone solves.  Bound: the FP32 dot product of two rows of Y = X - I/2 (norms at
most 1/2) errs by at most n 2^-24 / 4, and the epilogue adds a few roundings of values
below 1."""
import numpy as np
import pytest
import torch

from paper_2107_02737_gb300 import inputs
import paper_2107_02737_gb300.sp2 as sp2
from tests._gpu import dev, host

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [1, 129, 768, 769, 1500, 1537])
@pytest.mark.parametrize("choice", [0, 1])
def test_layer_at_tile_side_edges(n, choice):
    rng = np.random.default_rng(n)
    q, _ = np.linalg.qr(rng.standard_normal((n, n)))
    x = (q * rng.uniform(0.0, 1.0, n)) @ q.T
    x = np.float32((x + x.T) / 2)
    X, res = sp2.apply_layers(dev(x, torch.float32), [choice], precision="fp32")
    x = x.astype(np.float64)
    ref = x @ x if choice == 0 else 2.0 * x - x @ x
    got = host(X).astype(np.float64)
    assert np.array_equal(got, got.T)
    assert np.max(np.abs(got - ref)) <= (n + 32) * 2.0 ** -24 / 4
    assert abs(res.trace[1] - np.trace(got)) <= 1e-9 * n
    assert abs(res.trace_sq[1] - np.sum(got * got)) <= 1e-9 * n


def test_batch_of_mixed_tile_sides_equals_lone_solves():
    hams = [inputs.gapped_random(n, n // 2, inputs.rng_for(2, 800 + n)) for n in (200, 900, 1600)]
    Ds, res, status = sp2.density_batched([dev(h.H) for h in hams], [h.n_occ for h in hams], precision="fp32")
    assert status == sp2.OK
    for h, D, r in zip(hams, Ds, res):
        D1, r1 = sp2.density(dev(h.H), h.n_occ, precision="fp32")
        assert torch.equal(D, D1) and r.choices == r1.choices
