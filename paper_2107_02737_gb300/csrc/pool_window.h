// pool_window.h -- how much memory the calls' pool keeps: what the calls of the last two
// windows of POOL_WINDOW calls held at once at most, calls that ran side by side together.
#pragma once

#include <stddef.h>

#include <algorithm>

namespace sp2i {

constexpr int POOL_WINDOW = 12;   // so a large call's memory is back after at most 36 smaller ones

struct PoolWindow {
    size_t live = 0;          // held by the calls under way
    size_t peak[2] = {0, 0};  // most of it in this window and in the one before
    int calls = 0;

    // A call under way has taken `bytes`.
    void held(size_t bytes) {
        live += bytes;
        peak[0] = std::max(peak[0], live);
    }
    // A call that had taken `bytes` has ended; true at a window's end, with the bytes to keep.
    bool ended(size_t bytes, size_t &keep) {
        live -= bytes;
        if (++calls < POOL_WINDOW) return false;
        keep = std::max(peak[0], peak[1]);
        peak[1] = peak[0];
        peak[0] = live;
        calls = 0;
        return true;
    }
};

}  // namespace sp2i
