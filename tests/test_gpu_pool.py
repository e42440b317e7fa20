"""Workspaces that a call allocates come from a pool the library keeps between calls:
calls of mixed sizes from several threads and streams keep their results, and what a
large call needed goes back to the device once smaller calls have followed."""
import threading

import pytest
import torch

from paper_2107_02737_gb300 import inputs
import paper_2107_02737_gb300.sp2 as sp2
from tests._gpu import dev

pytestmark = pytest.mark.gpu


def test_threads_and_streams_share_the_pool():
    hams = [inputs.gapped_random(n, n // 2, inputs.rng_for(2, 40 + n)) for n in (96, 300, 520)]
    Hs = [dev(h.H) for h in hams]
    refs = [sp2.density(H, h.n_occ, precision="fp32")[0] for H, h in zip(Hs, hams)]
    torch.cuda.synchronize()
    wrong = []

    def work(k):
        stream = torch.cuda.Stream()
        with torch.cuda.stream(stream):
            for i in range(9):
                j = (i + k) % 3
                D, _ = sp2.density(Hs[j], hams[j].n_occ, precision="fp32", timeout_ms=20000.0)
                if not torch.equal(D, refs[j]):
                    wrong.append((k, i))

    threads = [threading.Thread(target=work, args=(k,)) for k in range(3)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not wrong


def test_memory_of_a_large_call_goes_back():
    n = 4096
    H = torch.diag(torch.linspace(-1.0, 1.0, n, device="cuda", dtype=torch.float64))
    small = dev(inputs.gapped_random(64, 32, inputs.rng_for(2, 9)).H)
    need = sp2.workspace_bytes(n)
    sp2.density(H, n // 2, max_layers=2)
    torch.cuda.synchronize()
    kept = torch.cuda.mem_get_info()[0]
    for _ in range(40):
        sp2.density(small, 32)
    torch.cuda.synchronize()
    assert torch.cuda.mem_get_info()[0] - kept >= need // 2
