"""How much the calls' memory pool keeps, on the CPU: the policy is plain C++, compiled here."""
import os
import subprocess

from paper_2107_02737_gb300 import build

PROGRAM = r"""
#include <cstdio>
#include "pool_window.h"
using sp2i::PoolWindow;
int main() {
    size_t keep = 0;
    PoolWindow w;
    // Pairs of calls side by side, 100 bytes each: both are kept for.
    for (int k = 0; k < sp2i::POOL_WINDOW; k += 2) {
        w.held(100);
        w.held(60);
        w.held(40);
        w.ended(100, keep);
        w.ended(100, keep);
    }
    printf("%zu\n", keep);
    // One window of small calls after them: the pair still counts; after two it does not.
    for (int r = 0; r < 2; ++r) {
        for (int k = 0; k < sp2i::POOL_WINDOW; ++k) {
            w.held(7);
            w.ended(7, keep);
        }
        printf("%zu\n", keep);
    }
    // A call that lasts over the end of a window counts in the next one too.
    w.held(500);
    for (int r = 0; r < 3; ++r) {
        for (int k = 0; k < sp2i::POOL_WINDOW; ++k) {
            w.held(7);
            w.ended(7, keep);
        }
    }
    printf("%zu %zu\n", keep, w.live);
}
"""


def test_pool_keeps_what_calls_side_by_side_need(tmp_path):
    src, exe = tmp_path / "window.cpp", tmp_path / "window"
    src.write_text(PROGRAM)
    subprocess.run(["g++", "-std=c++17", "-Wall", "-Werror", f"-I{build.CSRC}", str(src), "-o", str(exe)], check=True)
    out = subprocess.run([str(exe)], check=True, capture_output=True, text=True).stdout.split()
    assert out == ["200", "200", "7", "507", "500"]
    # The pool itself asks this policy, with every piece a call takes and the call's end.
    text = open(os.path.join(build.CSRC, "device_pool.cu")).read()
    assert "window.held(bytes)" in text and "window.ended(bytes, keep)" in text
