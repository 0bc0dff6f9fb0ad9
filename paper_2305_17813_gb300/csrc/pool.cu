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
// Bounds: the pool keeps what the library's objects hold (`kept` below; call
// workspaces do not count) and kPoolHold bytes beside it; what it has beyond
// that and nothing uses goes back to the device at the next synchronisation, at
// once when an object is destroyed, and all of it when an allocation fails
// (which is then tried once more) and on mk_trim.
// Threads and streams: the CUDA pool serialises its calls itself and hands a
// block freed in one stream to another only when the free has completed; the
// table below is behind a mutex.
#include "meerkat.h"
#include "pool.h"

#include <algorithm>
#include <mutex>

namespace {

// Below 1 % of the device, so that another allocator in the process hardly
// misses it, and enough for a graph of 33 M edges to be destroyed and made again
// without mapping; a larger one maps the rest anew.
constexpr uint64_t kPoolHold = 2ull << 30;
constexpr size_t kFollow = 1 << 20; // kept allocations that move the threshold
constexpr int kMaxDevices = 64;

struct DevicePool {
    cudaMemPool_t pool = nullptr;
    unsigned long long ctx = 0; // id of the context the pool belongs to
    uint64_t kept = 0;          // bytes that outlive the call which allocated them
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

// The current device's entry, its pool made on first use; locks g_mutex.
cudaError_t device_pool(DevicePool **out, std::unique_lock<std::mutex> &lock)
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
    lock = std::unique_lock<std::mutex>(g_mutex);
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
        d.kept = 0;
        uint64_t hold = kPoolHold;
        cudaMemPoolSetAttribute(pool, cudaMemPoolAttrReleaseThreshold, &hold);
    }
    *out = &d;
    return cudaSuccess;
}

// Adds to the kept bytes; with `follow` the pool's threshold goes with them.
void count_kept(uint64_t add, uint64_t take, bool follow)
{
    DevicePool *d = nullptr;
    std::unique_lock<std::mutex> lock;
    if (device_pool(&d, lock) != cudaSuccess)
        return;
    d->kept += add;
    d->kept -= std::min(d->kept, take);
    uint64_t most = d->kept + kPoolHold;
    if (follow)
        cudaMemPoolSetAttribute(d->pool, cudaMemPoolAttrReleaseThreshold, &most);
}

bool capturing(cudaStream_t s)
{
    cudaStreamCaptureStatus st = cudaStreamCaptureStatusNone;
    return cudaStreamIsCapturing(s, &st) != cudaSuccess || st != cudaStreamCaptureStatusNone;
}

} // namespace

namespace mk {

cudaError_t pool_alloc(void **p, size_t bytes, cudaStream_t s)
{
    *p = nullptr;
    cudaMemPool_t pool = nullptr;
    {
        DevicePool *d = nullptr;
        std::unique_lock<std::mutex> lock;
        const cudaError_t e = device_pool(&d, lock);
        if (e != cudaSuccess)
            return e;
        pool = d->pool;
    }
    cudaError_t e = cudaMallocFromPoolAsync(p, bytes ? bytes : 1, pool, s);
    if (e == cudaErrorMemoryAllocation) {
        cudaGetLastError();
        if (!capturing(s)) // a free is over when the host has seen its stream pass it
            cudaDeviceSynchronize();
        cudaMemPoolTrimTo(pool, 0);
        e = cudaMallocFromPoolAsync(p, bytes ? bytes : 1, pool, s);
    }
    if (e != cudaSuccess) {
        cudaGetLastError();
        *p = nullptr;
    }
    return e;
}

cudaError_t pool_alloc_kept(void **p, size_t bytes, cudaStream_t s)
{
    // memory allocated in a capture belongs to its graph
    cudaStreamCaptureStatus st = cudaStreamCaptureStatusNone;
    *p = nullptr;
    cudaError_t e = cudaStreamIsCapturing(s, &st);
    if (e != cudaSuccess)
        return e;
    if (st != cudaStreamCaptureStatusNone)
        return cudaErrorStreamCaptureUnsupported;
    if ((e = pool_alloc(p, bytes, s)) == cudaSuccess)
        count_kept(bytes, 0, bytes >= kFollow);
    return e;
}

cudaError_t pool_free(void *p, cudaStream_t s)
{
    return p ? cudaFreeAsync(p, s) : cudaSuccess;
}

cudaError_t pool_free_kept(void *p, size_t bytes, cudaStream_t s)
{
    if (!p)
        return cudaSuccess;
    const cudaError_t e = cudaFreeAsync(p, s);
    if (e == cudaSuccess)
        count_kept(0, bytes, bytes >= kFollow);
    return e;
}

cudaError_t pool_settle(uint64_t bytes)
{
    count_kept(0, bytes, true);
    return cudaSuccess;
}

} // namespace mk

extern "C" mk_status mk_trim(void)
{
    int dev = 0;
    // a free is over when the host has seen its stream pass it
    if (cudaGetDevice(&dev) != cudaSuccess || cudaDeviceSynchronize() != cudaSuccess)
        return MK_ERR_CUDA;
    std::lock_guard<std::mutex> lock(g_mutex);
    if (dev < 0 || dev >= kMaxDevices || !g_pools[dev].pool || g_pools[dev].ctx != context_id())
        return MK_OK;
    return cudaMemPoolTrimTo(g_pools[dev].pool, 0) == cudaSuccess ? MK_OK : MK_ERR_CUDA;
}
