// device_pool.cu -- a per-device memory pool for the calls' workspaces.
//
// Allocations from the default pool went back to the system at the end of every call
// (its release threshold is zero), and mapping them again took 0.2 ms of a call at
// N = 600 and 0.9 ms at N = 4096.  The library's own pool keeps what the latest
// calls needed, at most POOL_KEEP_MAX bytes: after every POOL_WINDOW calls it is trimmed
// to the largest call of the last two windows, and it is emptied when an allocation
// fails.  The pool is CUDA's own stream-ordered one, so blocks move between streams
// and threads only once their last use is ordered before the next.
#include "device_pool.h"

#include <algorithm>
#include <mutex>

namespace sp2i {

namespace {

constexpr size_t POOL_KEEP_MAX = (size_t)4 << 30;   // 1.5 % of the device's memory
constexpr int POOL_WINDOW = 12;   // so a large call's memory is back after at most 36 smaller ones
constexpr int POOL_DEVICES = 64;

struct DevicePool {
    cudaMemPool_t pool = nullptr;
    bool tried = false;
    int calls = 0;
    size_t peak[2] = {0, 0};   // largest call of this window and of the one before
};
std::mutex g_mu;
DevicePool g_pool[POOL_DEVICES];

// The current device's pool, made on first use; nullptr where there is none (the
// default pool then serves).
cudaMemPool_t pool_of_device() {
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= POOL_DEVICES) {
        cudaGetLastError();
        return nullptr;
    }
    std::lock_guard<std::mutex> lock(g_mu);
    DevicePool &p = g_pool[dev];
    if (!p.tried) {
        p.tried = true;
        cudaMemPoolProps props = {};
        props.allocType = cudaMemAllocationTypePinned;
        props.location.type = cudaMemLocationTypeDevice;
        props.location.id = dev;
        unsigned long long keep = POOL_KEEP_MAX;
        if (cudaMemPoolCreate(&p.pool, &props) != cudaSuccess) p.pool = nullptr;
        else if (cudaMemPoolSetAttribute(p.pool, cudaMemPoolAttrReleaseThreshold, &keep) != cudaSuccess) {
            cudaMemPoolDestroy(p.pool);
            p.pool = nullptr;
        }
        cudaGetLastError();
    }
    return p.pool;
}

// One call that held `bytes` has ended.
void pool_call_done(size_t bytes) {
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= POOL_DEVICES) {
        cudaGetLastError();
        return;
    }
    cudaMemPool_t pool = nullptr;
    size_t keep = 0;
    {
        std::lock_guard<std::mutex> lock(g_mu);
        DevicePool &p = g_pool[dev];
        p.peak[0] = std::max(p.peak[0], bytes);
        if (++p.calls < POOL_WINDOW) return;
        pool = p.pool;
        keep = std::max(p.peak[0], p.peak[1]);
        p.peak[1] = p.peak[0];
        p.peak[0] = 0;
        p.calls = 0;
    }
    if (pool && cudaMemPoolTrimTo(pool, std::min(keep + keep / 8, POOL_KEEP_MAX)) != cudaSuccess) cudaGetLastError();
}

}  // namespace

void pool_release() {
    cudaMemPool_t pool = pool_of_device();
    if (pool && cudaMemPoolTrimTo(pool, 0) != cudaSuccess) cudaGetLastError();
}

void *CallMemory::get(size_t bytes) {
    if (fail) return nullptr;
    if (bytes == 0) bytes = 256;
    void *q = nullptr;
    cudaMemPool_t pool = pool_of_device();
    cudaError_t e = pool ? cudaMallocFromPoolAsync(&q, bytes, pool, s) : cudaMallocAsync(&q, bytes, s);
    if (e != cudaSuccess && pool) {   // give back what the pool keeps and try once more
        cudaGetLastError();
        cudaStreamSynchronize(s);
        cudaMemPoolTrimTo(pool, 0);
        e = cudaMallocFromPoolAsync(&q, bytes, pool, s);
    }
    if (e != cudaSuccess) {
        cudaGetLastError();
        return nullptr;
    }
    ptrs.push_back(q);
    total += bytes;
    return q;
}

CallMemory::~CallMemory() {
    for (void *q : ptrs) cudaFreeAsync(q, s);
    cudaStreamSynchronize(s);
    if (!ptrs.empty()) pool_call_done(total);
}

}  // namespace sp2i
