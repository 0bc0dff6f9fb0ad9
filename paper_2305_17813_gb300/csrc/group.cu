// Grouping of a batch's edges by slab list: a counting pass gives every edge
// its rank among its list's edges, the lists get ranges of one array, and the
// edges are written there.  One 4-lane group then applies a whole list and
// owns it: repeats of a pair are found among the list's few edges, a chain is
// walked once for all of them, and free pairs are filled with plain stores.
//
// What large batches took before, and why: a hash set of the whole batch's pairs
// (one random atomic an edge into a table far larger than L2, 33 G/s against
// 128 G/s for the counters here, which stay in L2), a sort of each tile of
// 256 edges, and one chain walk and one 64-bit CAS an edge.  Smaller ones, whose
// table stays in L2, still do (hash_batch).
#include "group.h"
#include "mk_host.h"

#include <algorithm>

using namespace mk;

namespace {

constexpr uint32_t kBlock = 256, kPer = 4; // edges a thread

// Rank of every edge in its list.  Four edges a thread, so that the index
// gathers and the counter atomics of four edges are in flight together; the
// lists' first edges append them to the active lists (block-aggregated).
__global__ void __launch_bounds__(kBlock) k_group_count(GView g, const uint32_t *__restrict__ src,
                                                        const uint32_t *__restrict__ dst,
                                                        const uint32_t *__restrict__ w, uint64_t n, uint2 *slot,
                                                        uint32_t *__restrict__ lst, uint8_t *__restrict__ rank,
                                                        uint32_t *__restrict__ alist, uint32_t *ctr)
{
    __shared__ uint32_t s_warp[kBlock / 32], s_base;
    const uint64_t i0 = blockIdx.x * (uint64_t)(kBlock * kPer) + threadIdx.x;
    uint32_t L[kPer], s[kPer], d[kPer], r[kPer];
    uint2 vi[kPer];
    bool bad = false;
#pragma unroll
    for (uint32_t k = 0; k < kPer; ++k) {
        const uint64_t i = i0 + k * kBlock;
        s[k] = i < n ? __ldg(src + i) : kNil;
        d[k] = i < n ? __ldg(dst + i) : 0;
        const bool ok = s[k] < g.V && d[k] < g.V && !(w && i < n && __ldg(w + i) == 0);
        bad = bad || (i < n && !ok);
        L[k] = ok ? 0u : kNil;
    }
#pragma unroll
    for (uint32_t k = 0; k < kPer; ++k)
        vi[k] = L[k] != kNil ? __ldg(&g.vinfo[s[k]]) : make_uint2(0, 0);
#pragma unroll
    for (uint32_t k = 0; k < kPer; ++k) {
        r[k] = 1;
        if (L[k] != kNil) {
            L[k] = vi[k].x + bucket_of(d[k], vi[k].y);
            r[k] = atomicAdd(&slot[L[k]].x, 1u);
        }
    }
    uint32_t lead = 0;
#pragma unroll
    for (uint32_t k = 0; k < kPer; ++k) {
        const uint64_t i = i0 + k * kBlock;
        if (i < n) {
            lst[i] = L[k];
            rank[i] = (uint8_t)min(r[k], 255u);
        }
        lead += r[k] == 0;
    }
    if (__ballot_sync(kFull, bad) && lane_id() == 0)
        set_status(g.st, kErrInvalid);
    if (!alist)
        return;
    uint32_t incl = lead;
#pragma unroll
    for (uint32_t o = 1; o < 32; o <<= 1) {
        const uint32_t t = __shfl_up_sync(kFull, incl, o);
        if (lane_id() >= o)
            incl += t;
    }
    if (lane_id() == 31)
        s_warp[threadIdx.x >> 5] = incl;
    __syncthreads();
    if (threadIdx.x == 0) {
        uint32_t t = 0;
        for (uint32_t k = 0; k < kBlock / 32; ++k) {
            const uint32_t c = s_warp[k];
            s_warp[k] = t;
            t += c;
        }
        s_base = t ? atomicAdd(&ctr[kGroupActive], t) : 0u;
    }
    __syncthreads();
    uint32_t at = s_base + s_warp[threadIdx.x >> 5] + incl - lead;
#pragma unroll
    for (uint32_t k = 0; k < kPer; ++k)
        if (r[k] == 0)
            alist[at++] = L[k];
}

// Ranges of the entry array, one atomic a block on the cursor, so that the
// ranges follow the order of the lists up to the order of the blocks.  The
// range of a list with more than `most` edges starts as a free hash set.  Four
// lists a thread: a block waits for its chain (list, count, scan, cursor), so
// there are as few blocks as fill the chip once (2^20 edges: 12 us, 26 with
// one list a thread).
__global__ void __launch_bounds__(kBlock) k_group_place(const uint32_t *__restrict__ alist, uint32_t H, uint2 *slot,
                                                        uint2 *ent, uint32_t most, uint32_t *ctr)
{
    __shared__ uint32_t s_warp[kBlock / 32], s_base;
    const uint32_t n = alist ? __ldcg(&ctr[kGroupActive]) : H;
    for (uint64_t b = blockIdx.x * (uint64_t)(kBlock * kPer); b < n; b += (uint64_t)gridDim.x * (kBlock * kPer)) {
        const uint64_t k0 = b + (uint64_t)threadIdx.x * kPer;
        uint32_t L[kPer], c[kPer], sum = 0;
#pragma unroll
        for (uint32_t j = 0; j < kPer; ++j)
            L[j] = k0 + j < n ? (alist ? alist[k0 + j] : (uint32_t)(k0 + j)) : kNil;
#pragma unroll
        for (uint32_t j = 0; j < kPer; ++j)
            c[j] = L[j] != kNil ? slot[L[j]].x : 0;
#pragma unroll
        for (uint32_t j = 0; j < kPer; ++j)
            sum += c[j];
        uint32_t incl = sum;
#pragma unroll
        for (uint32_t o = 1; o < 32; o <<= 1) {
            const uint32_t t = __shfl_up_sync(kFull, incl, o);
            if (lane_id() >= o)
                incl += t;
        }
        if (lane_id() == 31)
            s_warp[threadIdx.x >> 5] = incl;
        __syncthreads();
        if (threadIdx.x == 0) {
            uint32_t t = 0;
            for (uint32_t j = 0; j < kBlock / 32; ++j) {
                const uint32_t x = s_warp[j];
                s_warp[j] = t;
                t += x;
            }
            s_base = t ? atomicAdd(&ctr[kGroupCursor], t) : 0u;
        }
        __syncthreads();
        uint32_t off = s_base + s_warp[threadIdx.x >> 5] + incl - sum;
#pragma unroll
        for (uint32_t j = 0; j < kPer; ++j) {
            if (c[j])
                slot[L[j]].y = off;
            for (uint32_t big = __ballot_sync(kFull, c[j] > most); big; big &= big - 1) {
                const uint32_t l = __ffs(big) - 1;
                const uint32_t o = __shfl_sync(kFull, off, l), m = __shfl_sync(kFull, c[j], l);
                for (uint32_t e = lane_id(); e < m; e += 32)
                    ent[o + e] = make_uint2(kNil, kNil);
            }
            off += c[j];
        }
        __syncthreads(); // s_warp and s_base are written again
    }
}

// Writes every edge of the lists [lo, hi) to its list's range.
__global__ void __launch_bounds__(kBlock) k_group_scatter(const uint32_t *__restrict__ dst, uint64_t n,
                                                          const uint2 *__restrict__ slot, uint32_t *lst,
                                                          const uint8_t *__restrict__ rank, uint2 *ent, uint32_t lo,
                                                          uint32_t hi, uint32_t most, uint32_t *many, uint32_t *ctr)
{
    const uint64_t i0 = blockIdx.x * (uint64_t)(kBlock * kPer) + threadIdx.x;
    uint32_t L[kPer];
    uint2 sl[kPer];
#pragma unroll
    for (uint32_t k = 0; k < kPer; ++k) {
        const uint64_t i = i0 + k * kBlock;
        L[k] = i < n ? lst[i] : kNil;
        if (L[k] < lo || L[k] >= hi) // a hash-set index is past every list
            L[k] = kNil;
    }
#pragma unroll
    for (uint32_t k = 0; k < kPer; ++k)
        sl[k] = L[k] != kNil ? __ldg(&slot[L[k]]) : make_uint2(0, 0);
#pragma unroll
    for (uint32_t k = 0; k < kPer; ++k) {
        const uint64_t i = i0 + k * kBlock;
        if (L[k] == kNil)
            continue;
        const uint32_t d = __ldg(dst + i), c = sl[k].x;
        if (c <= most) {
            ent[sl[k].y + rank[i]] = make_uint2(d, (uint32_t)i);
            continue;
        }
        many[__ldg(&ctr[kGroupActive]) + atomicAdd(&ctr[kGroupMany], 1u)] = (uint32_t)i;
        // open addressing with linear probing, at most half full (k_dedup)
        uint32_t *set = reinterpret_cast<uint32_t *>(ent + sl[k].y);
        uint32_t h = group_hash(d, 2 * c);
        for (uint32_t probe = 0; probe < 2 * c; ++probe) {
            const uint32_t j = atomicCAS(&set[h], kNil, (uint32_t)i);
            if (j == kNil || __ldg(dst + j) == d) {
                if (j != kNil && j > (uint32_t)i)
                    atomicMin(&set[h], (uint32_t)i);
                break;
            }
            h = h + 1 == 2 * c ? 0 : h + 1;
        }
        lst[i] = kSlotBit | (2 * sl[k].y + h);
    }
}

constexpr uint64_t kEdgeBytes = 8 + 4 + 4 + 1; // ent, lst, alist (and after it many), rank

// Bytes of the per-edge arrays for cap edges.  A list with many edges has
// kGroupMax + 1 at least, so the lists with edges and the edges of the lists
// with many are at most cap (1 + 1 / 32) together.
uint64_t edge_bytes(uint64_t cap) { return cap * kEdgeBytes + (cap / 32 + 16) * 4; }

} // namespace

namespace mk {

void group_release(GroupScratch &gs, uint64_t *bytes, cudaStream_t s)
{
    const uint64_t edges = gs.cap ? edge_bytes(gs.cap) : 0;
    const uint64_t lists = gs.slot ? (uint64_t)gs.lists * 8 + kGroupWords * 4 : 0;
    pool_free_kept(gs.ent, edges, s);
    pool_free_kept(gs.slot, lists, s);
    *bytes -= edges + lists;
    gs = GroupScratch{};
}

cudaError_t group_reserve(GroupScratch &gs, uint64_t n, uint32_t H, cudaStream_t s, uint64_t *bytes)
{
    cudaError_t e = cudaSuccess;
    if (!gs.slot) {
        const uint64_t size = (uint64_t)H * 8 + kGroupWords * 4;
        if ((e = pool_alloc_kept((void **)&gs.slot, size, s)) != cudaSuccess)
            return e;
        gs.lists = H;
        gs.ctr = reinterpret_cast<uint32_t *>(gs.slot + H);
        *bytes += size;
        if ((e = cudaMemsetAsync(gs.slot, 0, size, s)) != cudaSuccess)
            return e;
    }
    if (n <= gs.cap)
        return cudaSuccess;
    const uint64_t old = gs.cap, want = n <= kHashDelete ? kHashRoom * n : n;
    const uint64_t cap = (std::max<uint64_t>({want, 1024, old + old / 2}) + 15) & ~15ull;
    if ((e = cudaStreamSynchronize(s)) != cudaSuccess)
        return e;
    pool_free_kept(gs.ent, old ? edge_bytes(old) : 0, s);
    *bytes -= old ? edge_bytes(old) : 0;
    gs.ent = nullptr;
    gs.cap = 0;
    if ((e = pool_alloc_kept((void **)&gs.ent, edge_bytes(cap), s)) != cudaSuccess)
        return e;
    *bytes += edge_bytes(cap);
    gs.cap = cap;
    gs.lst = reinterpret_cast<uint32_t *>(gs.ent + cap);
    gs.alist = gs.lst + cap;
    gs.rank = reinterpret_cast<uint8_t *>(gs.alist + cap + cap / 32 + 16);
    return cudaSuccess;
}

cudaError_t group_batch(const GView &g, GroupScratch &gs, const uint32_t *src, const uint32_t *dst, const uint32_t *w,
                        uint64_t n, uint32_t most, cudaStream_t s, GroupView *gv, int *launches)
{
    const bool dense = group_dense(g.H, n);
    uint32_t *alist = dense ? nullptr : gs.alist;
    cudaError_t e = cudaMemsetAsync(gs.ctr, 0, kGroupWords * 4, s);
    if (e != cudaSuccess)
        return e;
    const uint32_t grid = grid_for((n + kPer - 1) / kPer, kBlock);
    k_group_count<<<grid, kBlock, 0, s>>>(g, src, dst, w, n, gs.slot, gs.lst, gs.rank, alist, gs.ctr);
    const uint64_t lists = dense ? g.H : n;
    k_group_place<<<std::min<uint32_t>(grid_for((lists + kPer - 1) / kPer, kBlock), num_sms() * 16), kBlock, 0, s>>>(
        alist, g.H, gs.slot, gs.ent, most, gs.ctr);
    // One pass for each 64 MB of entries: the range of lists a pass writes
    // stays in L2, where its 8-byte stores run at 190 G/s; over an array
    // beyond L2 they run at 33 G/s.
    const uint32_t passes = dense ? (uint32_t)((n * 8 + (64ull << 20) - 1) / (64ull << 20)) : 1u;
    for (uint32_t p = 0; p < passes; ++p)
        k_group_scatter<<<grid, kBlock, 0, s>>>(dst, n, gs.slot, gs.lst, gs.rank, gs.ent,
                                                (uint32_t)((uint64_t)g.H * p / passes),
                                                (uint32_t)((uint64_t)g.H * (p + 1) / passes), most, gs.alist, gs.ctr);
    *launches += 2 + (int)passes;
    *gv = {gs.slot, gs.ent, gs.lst, gs.alist, alist, gs.ctr, most};
    return cudaGetLastError();
}

} // namespace mk
