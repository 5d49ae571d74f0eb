// Device memory of targets and of their builds, from one stream-ordered pool
// per device.  A build makes about 25 allocations; through cudaMalloc and
// cudaFree each took 40-90 us (and every cudaFree waited for the device): with them
// a 131k-point target took 1.19 ms to build and 0.25 ms to close, with the pool
// 0.55 and 0.01.  When a build or a close returns, the pool keeps at most
// POOL_KEEP unused bytes; every allocation of the library that finds no memory
// first gives those back to the device and tries again.  The pool's own calls
// are safe from any thread.
//
// A closed target's memory may still be in use on any of the caller's streams
// (or by a graph that replays a search), so a close waits for the device, as
// cudaFree does, through cudaFree: every target owns one small plain
// allocation, its fence, and freeing that waits (30 ms of queued work: 30 ms).
// cudaDeviceSynchronize instead fails, and ruins the capture, while any
// thread captures a stream; cudaFree in relaxed mode does not.  The anchor, a
// plain allocation that is never freed, keeps the block that fences are carved
// from mapped: allocating and freeing a fence takes 2 + 2 us with it, 77 + 50
// without.
#include <mutex>

#include "pc_internal.h"

namespace {

constexpr uint64_t POOL_KEEP = 256ull << 20;
constexpr size_t ANCHOR_BYTES = 256;

struct Pool {
    bool made;
    cudaMemPool_t pool;   // null: the device has no pools (plain allocations then)
    cudaStream_t frees;   // memory whose last use is known to be over is freed here
    void* anchor;
};
std::mutex g_pool_mu;
Pool g_pools[64];

Pool* current_pool() {
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return nullptr;
    std::lock_guard<std::mutex> lk(g_pool_mu);
    Pool& p = g_pools[dev];
    if (p.made) return &p;
    p.made = true;
    cudaMemPoolProps props{};
    props.allocType = cudaMemAllocationTypePinned;
    props.location.type = cudaMemLocationTypeDevice;
    props.location.id = dev;
    uint64_t keep = POOL_KEEP;
    RelaxedCapture relaxed;
    if (cudaMalloc(&p.anchor, ANCHOR_BYTES) != cudaSuccess) cudaGetLastError();  // slower fences, nothing else
    if (cudaStreamCreateWithFlags(&p.frees, cudaStreamNonBlocking) != cudaSuccess ||
        cudaMemPoolCreate(&p.pool, &props) != cudaSuccess ||
        cudaMemPoolSetAttribute(p.pool, cudaMemPoolAttrReleaseThreshold, &keep) != cudaSuccess) {
        cudaGetLastError();
        p.pool = nullptr;
    }
    return &p;
}

// The pool's unused memory back to the device.
void give_back(Pool* p) {
    if (!p || !p->pool) return;
    RelaxedCapture relaxed;
    cudaStreamSynchronize(p->frees);
    cudaMemPoolTrimTo(p->pool, 0);
}

}  // namespace

cudaError_t pc_dev_alloc(void** out, size_t bytes, cudaStream_t s) {
    Pool* p = current_pool();
    if (!p) return cudaErrorInvalidDevice;
    if (!p->pool) return cudaMalloc(out, bytes);
    cudaError_t e = cudaMallocFromPoolAsync(out, bytes, p->pool, s);
    if (e == cudaErrorMemoryAllocation) {
        cudaGetLastError();
        cudaStreamSynchronize(s);
        give_back(p);
        e = cudaMallocFromPoolAsync(out, bytes, p->pool, s);
    }
    return e;
}

void pc_dev_free(void* ptr, cudaStream_t s) {
    Pool* p = current_pool();
    if (!ptr || !p) return;
    if (p->pool) cudaFreeAsync(ptr, s);
    else cudaFree(ptr);
}

cudaError_t pc_plain_alloc(void** out, size_t bytes) {
    cudaError_t e = cudaMalloc(out, bytes);
    if (e == cudaErrorMemoryAllocation) {
        cudaGetLastError();
        give_back(current_pool());
        e = cudaMalloc(out, bytes);
    }
    return e;
}

cudaError_t pc_fence_alloc(void** out, size_t bytes) {
    if (!current_pool()) return cudaErrorInvalidDevice;  // the anchor first
    RelaxedCapture relaxed;
    return pc_plain_alloc(out, bytes);
}

void pc_dev_free_idle(void* fence, void* const* ptrs, int n) {
    Pool* p = current_pool();
    if (!p || !fence) return;  // without a fence nothing else was allocated
    RelaxedCapture relaxed;
    if (cudaFree(fence) != cudaSuccess) {  // the context is lost, and the memory with it
        cudaGetLastError();
        return;
    }
    for (int i = 0; i < n; ++i) {
        if (!ptrs[i]) continue;
        if (p->pool) cudaFreeAsync(ptrs[i], p->frees);
        else cudaFree(ptrs[i]);
    }
    // The pool gives back what is above POOL_KEEP at a synchronisation, asked for
    // only then: on every close it cost the build of a 131k scan after it 45 us.
    uint64_t held = 0;
    if (p->pool && (cudaMemPoolGetAttribute(p->pool, cudaMemPoolAttrReservedMemCurrent, &held) != cudaSuccess ||
                    held > POOL_KEEP))
        cudaStreamSynchronize(p->frees);
}
