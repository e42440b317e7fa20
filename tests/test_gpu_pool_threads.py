"""Solves from several threads and streams at once, on the pool's memory: every one of them
ends, without an error, with the bits of the same solve alone.  FP32, and FP16 in single-CTA
tiles (cooperative launches, whose CTAs are resident together or not at all)."""
import threading

import pytest
import torch

from paper_2107_02737_gb300 import inputs
import paper_2107_02737_gb300.sp2 as sp2
from tests._gpu import dev

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", ["fp32", "fp16"])
def test_every_solve_of_every_thread_ends_well(precision):
    hams = [inputs.gapped_random(n, n // 2, inputs.rng_for(2, 40 + n)) for n in (96, 300, 520)]
    Hs = [dev(h.H) for h in hams]
    refs = [sp2.density(H, h.n_occ, precision=precision)[0] for H, h in zip(Hs, hams)]
    torch.cuda.synchronize()
    done, wrong = [], []

    def work(k):
        try:
            stream = torch.cuda.Stream()
            with torch.cuda.stream(stream):
                for i in range(15):   # past the end of the pool's window of calls, three times over
                    j = (i + k) % 3
                    D, res = sp2.density(Hs[j], hams[j].n_occ, precision=precision, timeout_ms=20000.0)
                    assert res.converged and res.cta_group == (0 if precision == "fp32" else 1)
                    if not torch.equal(D, refs[j]):
                        wrong.append((k, i))
                    done.append((k, i))
        except BaseException as e:   # a thread's exception does not reach the test by itself
            wrong.append((k, repr(e)))

    threads = [threading.Thread(target=work, args=(k,)) for k in range(3)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not wrong
    assert len(done) == 45
