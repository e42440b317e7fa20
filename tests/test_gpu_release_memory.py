"""sp2_release_memory: what the calls' pool keeps goes back to the device when asked for, and
later calls are served as before."""
import pytest
import torch

import paper_2107_02737_gb300.sp2 as sp2

pytestmark = pytest.mark.gpu


def test_kept_memory_goes_back_on_request():
    n = 4096
    H = torch.diag(torch.linspace(-1.0, 1.0, n, device="cuda", dtype=torch.float64))
    need = sp2.workspace_bytes(n)
    D0, _ = sp2.density(H, n // 2, max_layers=2)
    torch.cuda.synchronize()
    kept = torch.cuda.mem_get_info()[0]
    sp2.release_memory()
    assert torch.cuda.mem_get_info()[0] - kept >= need // 2
    sp2.release_memory()
    D1, _ = sp2.density(H, n // 2, max_layers=2)
    assert torch.equal(D0, D1)
