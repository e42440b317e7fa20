"""A batch whose completions stop coming: CTA 0 withholds the first one (test_hook = 1), the
waits of the batch schedule (for an instance's decision, and of the warp that decides) run
out after timeout_ms, and the call returns SP2_ERR_TIMEOUT with the context usable.  Short
limits run out while the other instances are still in the middle of their chains."""
import ctypes

import pytest
import torch

from paper_2107_02737_gb300 import inputs
import paper_2107_02737_gb300.sp2 as sp2
from tests._gpu import dev

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("cta_group", [0, 1, 2])
@pytest.mark.parametrize("timeout_ms", [1.0, 50.0])
def test_batch_wait_runs_out(cta_group, timeout_ms):
    sizes = [1300, 700, 256, 256, 130, 640]
    hams = [inputs.gapped_random(n, n // 2, inputs.rng_for(2, 60 + i)) for i, n in enumerate(sizes)]
    Hs = [dev(h.H) for h in hams]
    Ds = [torch.empty((n, n), dtype=torch.float32, device="cuda") for n in sizes]
    B = len(sizes)
    o = sp2.make_opts("bf16", timeout_ms=timeout_ms, cta_group=cta_group)
    o.test_hook = 1
    hp = (ctypes.c_void_p * B)(*[h.data_ptr() for h in Hs])
    dp = (ctypes.c_void_p * B)(*[d.data_ptr() for d in Ds])
    nn = (ctypes.c_int * B)(*sizes)
    occ = (ctypes.c_double * B)(*[float(h.n_occ) for h in hams])
    for _ in range(3):
        s = sp2.load().sp2_density_batched(B, hp, nn, occ, 1e-6, dp, None, ctypes.byref(o), None, 0,
                                           ctypes.c_void_p(torch.cuda.current_stream().cuda_stream))
        assert s == sp2.ERR_TIMEOUT
    Ds, res, status = sp2.density_batched(Hs, [h.n_occ for h in hams], precision="bf16", cta_group=cta_group)
    assert status == sp2.OK
    D1, r1 = sp2.density(Hs[1], hams[1].n_occ, precision="bf16", cta_group=cta_group)
    assert torch.equal(Ds[1], D1) and res[1].trace == r1.trace
