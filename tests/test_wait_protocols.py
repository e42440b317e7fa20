"""Waits of the persistent kernels, by their source text: how a warp's or a CTA's threads
come to act on what one of them waited for.  (A fault here would hang or race on the GPU,
so it is not provoked there.)"""
import os
import re

from paper_2107_02737_gb300 import build


def source(name):
    text = open(os.path.join(build.CSRC, name)).read()
    return re.sub(r"//[^\n]*", "", text)


def block(text, start):
    """The brace block that opens at or after `start`."""
    i = text.index("{", start)
    depth = 0
    for j in range(i, len(text)):
        depth += {"{": 1, "}": -1}.get(text[j], 0)
        if depth == 0:
            return text[i:j + 1]
    raise AssertionError("unbalanced braces")


def test_batch_epilogue_warps_take_a_decision_together():
    """The eight epilogue warps meet at named barriers inside a tile's epilogue, so either
    all of them take a list entry or none does: one thread waits for the entry's decision,
    and a barrier of all eight lies between that wait and the tile."""
    batch = block(source("tc_kernel.cu"), source("tc_kernel.cu").index("if constexpr (SCHED == RUN_BATCH) {"))
    epi = block(batch, batch.index("else if (warp < 2 + EPI_WARPS)"))
    calls = [m.start() for m in re.finditer(r"flow_wait_instance\(", epi)]
    assert len(calls) == 1
    guard = epi.index("if (ew == 0 && lane == 0)")
    assert guard < calls[0] < guard + len(block(epi, guard)) + len("if (ew == 0 && lane == 0) ")
    after = epi[calls[0]:epi.index("epilogue_tile(w)")]
    assert "bar.sync 1" in after
    # what the warps branch on is what the barrier handed over, nothing of their own
    assert "*abort" not in after and "__shfl" not in after


def test_a_warp_acts_on_lane_0s_wait_only_after_a_warp_barrier():
    """A shuffle hands a value on but orders no memory: where the value is what lane 0
    waited for, it goes through warp_waited, which adds the __syncwarp."""
    waits = r"mbar_wait|flow_wait|flow_wait_instance|ld_acquire"
    seen = 0
    for name in ("tc_ptx.cuh", "tc_kernel.cu", "exact_kernel.cu", "simt_kernel.cu"):
        text = source(name)
        for m in re.finditer(r"(__shfl_sync\(0xffffffffu, (\w+), 0\)|warp_waited\((\w+)\))", text):
            var = m.group(2) or m.group(3)
            assigned = re.findall(r"\b%s = ([^;]*);" % var, text[:m.start()])
            if assigned and re.search(r"\b(%s)\(" % waits, assigned[-1]):
                seen += 1
                assert m.group(3), f"{name}: {assigned[-1]}"
    assert seen >= 7
    helper = block(source("device_common.cuh"), source("device_common.cuh").index("int warp_waited(int lane0)"))
    assert helper.index("__shfl_sync") < helper.index("__syncwarp")


def test_a_stopped_wait_looks_at_its_counter_once_more():
    """The CTA of a pair that first sees the last layer complete ends the other one, which
    must not take that for a failure of its own wait: CTA 0 writes the last decision."""
    text = source("tc_kernel.cu")
    body = block(text, text.index("bool flow_wait(const RunParams &p, const unsigned int *counter"))
    stop = block(body, body.index("if (*abort || ld_volatile(p.err) != 0)"))
    assert "return" not in stop and "fence.acq_rel.cluster" in stop and "break" in stop
    assert body.rstrip().endswith("return ld_acquire(counter) >= target;\n}")
    halt = block(text, text.index("void tc_abort(RoundCtl &rc"))
    assert halt.index("fence.acq_rel.cluster") < halt.index("st.shared::cluster")
