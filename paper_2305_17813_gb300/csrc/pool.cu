// Device memory of the library: one CUDA memory pool a device, its own (the
// process's default pool and its settings are left alone).
//
// Why: a graph of 33 M edges holds 1.8 GB, and mapping and unmapping that much
// costs 0.8 ms a GB with cudaMalloc / cudaFree -- creating and destroying the
// graph took longer than filling it (2.9 of a load's 5.9 ms; 0.1 from a pool
// that still holds the memory of the graph before).  The call workspaces,
// which came from the default pool and were unmapped at every synchronisation,
// come from here too.
//
// Bounds: the pool gives memory that nothing uses back to the device down to
// kPoolHold bytes at the next synchronisation (its release threshold counts
// the memory in use too and follows it), all of it when an allocation fails
// (which is then tried once more) and on mk_trim.
// Threads and streams: the CUDA pool serialises its calls itself and hands a
// block freed in one stream to another only when the free has completed; the
// table below is behind a mutex.
#include "mk_host.h"

#include <mutex>

namespace {

constexpr uint64_t kPoolHold = 2ull << 30;
constexpr size_t kFollow = 1 << 20; // allocations that move the threshold
constexpr int kMaxDevices = 64;

struct DevicePool {
    cudaMemPool_t pool = nullptr;
    unsigned long long ctx = 0; // id of the context the pool belongs to
};
std::mutex g_mutex;
DevicePool g_pools[kMaxDevices];

typedef int (*CtxGetIdFn)(void *ctx, unsigned long long *id);

// Id of the calling thread's current context (a cudaDeviceReset starts a new
// one, and ends the pools of the old); 0 if it cannot be had.
unsigned long long context_id()
{
    static const CtxGetIdFn fn = [] {
        void *p = nullptr;
        cudaDriverEntryPointQueryResult q = cudaDriverEntryPointSymbolNotFound;
        if (cudaGetDriverEntryPointByVersion("cuCtxGetId", &p, 12000, cudaEnableDefault, &q) != cudaSuccess ||
            q != cudaDriverEntryPointSuccess)
            p = nullptr;
        cudaGetLastError();
        return (CtxGetIdFn)p;
    }();
    unsigned long long id = 0;
    return fn && fn(nullptr, &id) == 0 ? id : 0;
}

cudaError_t device_pool(cudaMemPool_t *out)
{
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess)
        return e;
    if (dev < 0 || dev >= kMaxDevices)
        return cudaErrorInvalidDevice;
    unsigned long long ctx = context_id();
    if (!ctx) { // no context yet on this thread
        cudaFree(nullptr);
        ctx = context_id();
    }
    std::lock_guard<std::mutex> lock(g_mutex);
    DevicePool &d = g_pools[dev];
    if (!d.pool || d.ctx != ctx) {
        cudaMemPoolProps props{};
        props.allocType = cudaMemAllocationTypePinned;
        props.location.type = cudaMemLocationTypeDevice;
        props.location.id = dev;
        cudaMemPool_t pool = nullptr;
        if ((e = cudaMemPoolCreate(&pool, &props)) != cudaSuccess)
            return e;
        d.pool = pool;
        d.ctx = ctx;
    }
    *out = d.pool;
    return cudaSuccess;
}

// The threshold: what is in use and kPoolHold.
void follow_use(cudaMemPool_t pool)
{
    uint64_t used = 0;
    if (cudaMemPoolGetAttribute(pool, cudaMemPoolAttrUsedMemCurrent, &used) != cudaSuccess)
        return;
    used += kPoolHold;
    cudaMemPoolSetAttribute(pool, cudaMemPoolAttrReleaseThreshold, &used);
}

} // namespace

namespace mk {

cudaError_t pool_alloc(void **p, size_t bytes, cudaStream_t s)
{
    *p = nullptr;
    cudaMemPool_t pool = nullptr;
    cudaError_t e = device_pool(&pool);
    if (e != cudaSuccess)
        return e;
    e = cudaMallocFromPoolAsync(p, bytes ? bytes : 1, pool, s);
    if (e == cudaErrorMemoryAllocation) {
        cudaGetLastError();
        cudaMemPoolTrimTo(pool, 0);
        e = cudaMallocFromPoolAsync(p, bytes ? bytes : 1, pool, s);
    }
    if (e != cudaSuccess) {
        cudaGetLastError();
        *p = nullptr;
    } else if (bytes >= kFollow) {
        follow_use(pool);
    }
    return e;
}

void pool_settle()
{
    cudaMemPool_t pool = nullptr;
    if (device_pool(&pool) == cudaSuccess)
        follow_use(pool);
}

cudaError_t pool_alloc_kept(void **p, size_t bytes, cudaStream_t s)
{
    // memory allocated in a capture belongs to its graph
    cudaStreamCaptureStatus st = cudaStreamCaptureStatusNone;
    *p = nullptr;
    const cudaError_t e = cudaStreamIsCapturing(s, &st);
    if (e != cudaSuccess)
        return e;
    return st == cudaStreamCaptureStatusNone ? pool_alloc(p, bytes, s) : cudaErrorStreamCaptureUnsupported;
}

void pool_free(void *p, cudaStream_t s)
{
    if (p)
        cudaFreeAsync(p, s);
}

} // namespace mk

extern "C" mk_status mk_trim(void)
{
    int dev = 0;
    MK_CUDA(cudaGetDevice(&dev));
    MK_CUDA(cudaDeviceSynchronize()); // a free is over when the host has seen its stream pass it
    std::lock_guard<std::mutex> lock(g_mutex);
    if (dev < 0 || dev >= kMaxDevices || !g_pools[dev].pool || g_pools[dev].ctx != context_id())
        return MK_OK;
    MK_CUDA(cudaMemPoolTrimTo(g_pools[dev].pool, 0));
    return MK_OK;
}
