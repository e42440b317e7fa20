"""A CTA pair that never becomes resident (test_hook = 3: CTA 0 of a pair launch withholds a
completion), at sizes whose tiles the library takes in pairs: 256 x 128 and 256 x 256 in one
wave, 256 x 256 in several, and the rounds of a response.  Left to itself the call waits out
timeout_ms, retries with single-CTA tiles and succeeds; forced to pairs it reports the
timeout."""
import ctypes
import time

import pytest
import torch

import paper_2107_02737_gb300.sp2 as sp2

pytestmark = pytest.mark.gpu
TIMEOUT_MS = 100.0


def diagonal_system(n):
    lam = torch.cat([torch.linspace(-1.0, -0.1, n // 2), torch.linspace(0.1, 1.0, n - n // 2)]).double()
    g = torch.Generator().manual_seed(n)
    return torch.diag(lam[torch.randperm(n, generator=g)]).cuda()


def options(cta_group=0, hook=3):
    o = sp2.make_opts("fp16", timeout_ms=TIMEOUT_MS, cta_group=cta_group)
    o.test_hook = hook
    return o


def call(name, H, o, *outs, M=None):
    st = sp2._new_stats()
    args = [ctypes.c_void_p(t.data_ptr()) for t in ([H] if M is None else [H, M])]
    extra = [] if M is None else [None]   # no earlier forward run to replay
    torch.cuda.synchronize()
    t0 = time.perf_counter()
    s = getattr(sp2.load(), name)(*args, H.shape[0], float(H.shape[0] // 2), 1e-6, *extra,
                                  *[ctypes.c_void_p(t.data_ptr()) for t in outs], ctypes.byref(st), ctypes.byref(o),
                                  None, 0, ctypes.c_void_p(torch.cuda.current_stream().cuda_stream))
    return s, st, 1e3 * (time.perf_counter() - t0)


@pytest.mark.parametrize("n", [1409, 1537, 2304, 4096])
def test_density_retries_with_single_ctas(n):
    H = diagonal_system(n)
    D = torch.empty((n, n), dtype=torch.float32, device="cuda")
    s, st, ms = call("sp2_density", H, options(hook=0), D)
    assert s == sp2.OK and st.cta_group == 2   # pairs, without the hook
    s, st, ms = call("sp2_density", H, options(), D)
    assert s == sp2.OK and st.cta_group == 1 and ms >= TIMEOUT_MS
    ref, _ = sp2.density(H, n // 2, cta_group=1)
    assert torch.equal(D, ref)
    s, _, ms = call("sp2_density", H, options(cta_group=2), D)
    assert s == sp2.ERR_TIMEOUT and ms >= TIMEOUT_MS


@pytest.mark.parametrize("n", [1300, 1600])
def test_response_retries_with_single_ctas(n):
    H = diagonal_system(n)
    M = torch.full_like(H, 0.01)
    D, D1 = (torch.empty((n, n), dtype=torch.float32, device="cuda") for _ in range(2))
    s, st, _ = call("sp2_response", H, options(hook=0), D, D1, M=M)
    assert s == sp2.OK and st.cta_group == 2
    s, st, ms = call("sp2_response", H, options(), D, D1, M=M)
    assert s == sp2.OK and st.cta_group == 1 and ms >= TIMEOUT_MS
    _, ref, _ = sp2.response(H, M, n // 2, cta_group=1)
    assert torch.equal(D1, ref)
