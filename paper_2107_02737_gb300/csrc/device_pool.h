// device_pool.h -- device memory of one call's workspace and staging buffers.
#pragma once

#include <cuda_runtime.h>
#include <stddef.h>

#include <vector>

namespace sp2i {

// Device allocations owned by one call, stream-ordered on `s`, freed and the stream
// waited for on every exit path.  With `fail` set (sp2_opts.test_hook = 2, host-side
// fault injection) every allocation reports failure, as an exhausted device would.
struct CallMemory {
    std::vector<void *> ptrs;
    cudaStream_t s;
    size_t total = 0;
    bool fail = false;
    explicit CallMemory(cudaStream_t st) : s(st) {}
    CallMemory(const CallMemory &) = delete;
    CallMemory &operator=(const CallMemory &) = delete;
    void *get(size_t bytes);   // nullptr when there is none
    ~CallMemory();
};

// Gives what the current device's pool keeps, and nothing uses, back to the device.
cudaError_t pool_release();

}  // namespace sp2i
