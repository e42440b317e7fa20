// device_pool.cu -- a per-device memory pool for the calls' workspaces.
//
// Allocations from the default pool went back to the system at the end of every call
// (its release threshold is zero), and mapping them again took 0.2 ms of a call at
// N = 600 and 0.9 ms at N = 4096.  The library's own pool keeps what the latest
// calls needed, at most POOL_KEEP_MAX bytes: after every POOL_WINDOW calls it is trimmed
// to what the calls of the last two windows held at once (PoolWindow), and it is emptied
// when an allocation fails.  The pool is CUDA's own stream-ordered one, so blocks move between streams
// and threads only once their last use is ordered before the next.
#include "device_pool.h"

#include <algorithm>
#include <mutex>

#include "pool_window.h"

namespace sp2i {

namespace {

constexpr size_t POOL_KEEP_MAX = (size_t)4 << 30;   // 1.5 % of the device's memory
constexpr int POOL_DEVICES = 64;

struct DevicePool {
    cudaMemPool_t pool = nullptr;
    bool tried = false;
    PoolWindow window;
};
std::mutex g_mu;
DevicePool g_pool[POOL_DEVICES];

// The current device's entry, nullptr where there is none.
DevicePool *pool_entry(int &dev) {
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= POOL_DEVICES) {
        cudaGetLastError();
        return nullptr;
    }
    return &g_pool[dev];
}

// The current device's pool, made on first use; nullptr where there is none (the
// default pool then serves).
cudaMemPool_t pool_of_device() {
    int dev = 0;
    DevicePool *entry = pool_entry(dev);
    if (!entry) return nullptr;
    std::lock_guard<std::mutex> lock(g_mu);
    DevicePool &p = *entry;
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

// A call under way has taken `bytes`.
void pool_held(size_t bytes) {
    int dev = 0;
    DevicePool *p = pool_entry(dev);
    if (!p) return;
    std::lock_guard<std::mutex> lock(g_mu);
    p->window.held(bytes);
}

// A call that had taken `bytes` has ended.
void pool_call_done(size_t bytes) {
    int dev = 0;
    DevicePool *p = pool_entry(dev);
    if (!p) return;
    cudaMemPool_t pool = nullptr;
    size_t keep = 0;
    {
        std::lock_guard<std::mutex> lock(g_mu);
        if (!p->window.ended(bytes, keep)) return;
        pool = p->pool;
    }
    if (pool && cudaMemPoolTrimTo(pool, std::min(keep + keep / 8, POOL_KEEP_MAX)) != cudaSuccess) cudaGetLastError();
}

}  // namespace

cudaError_t pool_release() {
    int dev = 0;
    DevicePool *p = pool_entry(dev);
    if (!p) return cudaErrorInvalidDevice;
    cudaMemPool_t pool = nullptr;
    {
        std::lock_guard<std::mutex> lock(g_mu);
        pool = p->pool;
    }
    const cudaError_t e = pool ? cudaMemPoolTrimTo(pool, 0) : cudaSuccess;
    if (e != cudaSuccess) cudaGetLastError();
    return e;
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
    pool_held(bytes);
    return q;
}

CallMemory::~CallMemory() {
    for (void *q : ptrs) cudaFreeAsync(q, s);
    cudaStreamSynchronize(s);
    if (!ptrs.empty()) pool_call_done(total);
}

}  // namespace sp2i
