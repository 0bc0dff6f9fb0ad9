"""The library's memory pool (csrc/pool.cu) against a model of the CUDA
runtime's stream-ordered pools, on the CPU: what the pool holds beside the
library's objects stays within its bound whatever the call workspaces were,
and an allocation that fails at first takes what is free."""
import ctypes
import os
import shutil
import subprocess

import pytest

from paper_2305_17813_gb300 import build

GB = 1 << 30
HOLD = 2 * GB

MODEL = r"""
// Two devices.  A freed block is free from the next synchronisation of its
// device on, which also releases free memory beyond the pool's threshold.
#include "pool.h"
#include "meerkat.h"
#include <cuda_runtime_api.h>
#include <algorithm>
#include <map>
typedef unsigned long long u64;
struct Dev { u64 used = 0, pending = 0, spare = 0, threshold = 0, room = 16ull << 30; bool capturing = false; };
static Dev devs[2];
static int cur = 0, wrong = 0, syncs[2];
static u64 next_ptr = 4096;
struct Block { int dev; u64 bytes; };
static std::map<u64, Block> blocks;
static Dev &dev_of(cudaMemPool_t p) { return devs[(u64)p - 1]; }
static void synced(int d)
{
    Dev &x = devs[d];
    ++syncs[d];
    x.spare += x.pending;
    x.pending = 0;
    const u64 held = x.used + x.spare;
    x.spare -= std::min(x.spare, held > x.threshold ? held - x.threshold : 0);
}
static int ctx_id(void *, u64 *id) { *id = 100 + cur; return 0; }
extern "C" {
cudaError_t cudaGetDevice(int *d) { *d = cur; return cudaSuccess; }
cudaError_t cudaSetDevice(int d) { cur = d; return cudaSuccess; }
cudaError_t cudaFree(void *) { return cudaSuccess; }
cudaError_t cudaGetLastError() { return cudaSuccess; }
cudaError_t cudaDeviceSynchronize() { synced(cur); return cudaSuccess; }
cudaError_t cudaStreamSynchronize(cudaStream_t) { synced(cur); return cudaSuccess; }
cudaError_t cudaStreamIsCapturing(cudaStream_t, cudaStreamCaptureStatus *s)
{
    *s = devs[cur].capturing ? cudaStreamCaptureStatusActive : cudaStreamCaptureStatusNone;
    return cudaSuccess;
}
cudaError_t cudaGetDriverEntryPointByVersion(const char *, void **f, unsigned int, unsigned long long,
                                             cudaDriverEntryPointQueryResult *r)
{
    *f = (void *)ctx_id;
    *r = cudaDriverEntryPointSuccess;
    return cudaSuccess;
}
cudaError_t cudaMemPoolCreate(cudaMemPool_t *p, const cudaMemPoolProps *props)
{
    *p = (cudaMemPool_t)(u64)(props->location.id + 1);
    return cudaSuccess;
}
cudaError_t cudaMemPoolSetAttribute(cudaMemPool_t p, cudaMemPoolAttr, void *v)
{
    dev_of(p).threshold = *(u64 *)v;
    return cudaSuccess;
}
cudaError_t cudaMemPoolGetAttribute(cudaMemPool_t p, cudaMemPoolAttr, void *v)
{
    *(u64 *)v = dev_of(p).used;
    return cudaSuccess;
}
cudaError_t cudaMemPoolTrimTo(cudaMemPool_t p, size_t) { dev_of(p).spare = 0; return cudaSuccess; }
cudaError_t cudaMallocFromPoolAsync(void **out, size_t n, cudaMemPool_t p, cudaStream_t)
{
    Dev &x = dev_of(p);
    const u64 more = n > x.spare ? n - x.spare : 0;
    if (x.used + x.pending + x.spare + more > x.room)
        return cudaErrorMemoryAllocation;
    x.spare = x.spare + more - n;
    x.used += n;
    *out = (void *)next_ptr;
    blocks[next_ptr] = {(int)((u64)p - 1), n};
    next_ptr += 4096;
    return cudaSuccess;
}
cudaError_t cudaFreeAsync(void *p, cudaStream_t)
{
    const Block b = blocks.at((u64)p);
    blocks.erase((u64)p);
    wrong += b.dev != cur;
    devs[b.dev].used -= b.bytes;
    devs[b.dev].pending += b.bytes;
    return cudaSuccess;
}

u64 t_alloc(u64 n, int kept)
{
    void *p = nullptr;
    const cudaError_t e = kept ? mk::pool_alloc_kept(&p, n, nullptr) : mk::pool_alloc(&p, n, nullptr);
    return e == cudaSuccess ? (u64)p : 0;
}
void t_free(u64 p, u64 kept) { kept ? mk::pool_free_kept((void *)p, kept, nullptr) : mk::pool_free((void *)p, nullptr); }
void t_settle(u64 n) { mk::pool_settle(n); }
void t_destroy(int dev, u64 p, u64 kept) // as the stores' destroy calls do
{
    mk::DeviceScope on(dev);
    cudaDeviceSynchronize();
    mk::pool_free((void *)p, nullptr);
    mk::pool_settle(kept);
}
void t_sync() { synced(cur); }
void t_device(int d) { cur = d; }
int t_current() { return cur; }
void t_capture(int on) { devs[cur].capturing = on; }
int t_wrong() { return wrong; }
int t_syncs(int d) { return syncs[d]; }
u64 t_held(int d) { return devs[d].used + devs[d].pending + devs[d].spare; }
u64 t_threshold(int d) { return devs[d].threshold; }
}
"""


@pytest.fixture()
def pool(tmp_path):
    """A fresh copy of the pool and of the model."""
    src = tmp_path / "model.cpp"
    src.write_text(MODEL)
    lib = tmp_path / "libpool.so"
    cuda = os.path.join(os.path.dirname(os.path.dirname(os.path.realpath(build.nvcc()))), "include")
    subprocess.run([shutil.which("g++") or "g++", "-std=c++17", "-shared", "-fPIC", "-I", build.CSRC, "-I", build.INCLUDE,
                    "-I", cuda, "-x", "c++", os.path.join(build.CSRC, "pool.cu"), str(src), "-o", str(lib)], check=True)
    x = ctypes.CDLL(str(lib))
    for f in ("t_alloc", "t_held", "t_threshold"):
        getattr(x, f).restype = ctypes.c_uint64
    x.t_alloc.argtypes = [ctypes.c_uint64, ctypes.c_int]
    x.t_free.argtypes = [ctypes.c_uint64, ctypes.c_uint64]
    x.t_settle.argtypes = [ctypes.c_uint64]
    x.t_destroy.argtypes = [ctypes.c_int, ctypes.c_uint64, ctypes.c_uint64]
    return x


def test_workspaces_do_not_count_as_kept(pool):
    graph = pool.t_alloc(1 * GB, 1)
    assert graph and pool.t_threshold(0) == 1 * GB + HOLD
    for big in (3 * GB, 9 * GB, 5 * GB):  # a call's work arrays, freed in the call
        a, b = pool.t_alloc(big, 0), pool.t_alloc(GB // 2, 0)
        assert a and b
        pool.t_free(a, 0)
        pool.t_free(b, 0)
        pool.t_sync()
        assert pool.t_held(0) <= 1 * GB + HOLD
    old, new = pool.t_alloc(1 * GB, 1), pool.t_alloc(4 * GB, 1)  # an array regrown
    pool.t_free(old, 1 * GB)
    pool.t_sync()
    assert pool.t_threshold(0) == 5 * GB + HOLD
    pool.t_free(new, 0)  # destroyed: freed without their sizes, which settle takes off
    pool.t_free(graph, 0)
    pool.t_settle(5 * GB)
    pool.t_sync()
    assert pool.t_threshold(0) == HOLD and pool.t_held(0) <= HOLD


def test_a_failed_allocation_takes_what_is_free(pool):
    a = pool.t_alloc(12 * GB, 1)
    pool.t_free(a, 12 * GB)  # still on its way: no one has waited for its stream
    assert pool.t_alloc(14 * GB, 1)
    assert pool.t_alloc(4 * GB, 0) == 0


def test_kept_allocations_are_refused_in_a_capture(pool):
    pool.t_capture(1)
    assert pool.t_alloc(GB, 1) == 0
    assert pool.t_alloc(GB, 0)
    pool.t_capture(0)
    assert pool.t_alloc(GB, 1)
