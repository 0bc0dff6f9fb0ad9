// Graph analytics on the slab store beyond BFS/SSSP/WCC: PageRank (paper,
// Sec. "Dynamic PageRank", Algorithm "Page Rank - Static / Incremental /
// Decremental", Eq. 1) and triangle counting (paper, Sec. "Dynamic Triangle
// Counting", Algorithms "Triangle Counting - Incremental / Decremental" and
// the Count kernel).
//
// PageRank.  The paper's Compute kernel pulls over a graph object that
// stores in-edges; this store keeps out-edges.  A call first copies its live
// edges out of the slabs into bins by destination, so that each super-step
// reads them in order and adds u's contribution PR[u] / out[u] up in shared
// memory for every edge u -> v of a bin (the idea of propagation blocking:
// Beamer, Asanovic and Patterson, "Reducing Pagerank Communication via
// Propagation Blocking", IPDPS 2017; here the edges are binned, once a call, not
// the contributions of each step).  Graphs and calls for which the copy
// does not pay (more than 2^24 vertices, fewer than four super-steps, no
// memory for it) push along the slabs instead, in address order.  Ranks,
// contributions and sums are 64-bit fixed-point numbers (value * 2^48) added
// as integers, so a result does not depend on the order of the additions, nor
// on which of the two forms runs; the L1 delta of a super-step is summed the
// same way.  The teleport term for zero-out-degree vertices is added as in
// the paper (FindTeleportProb).  The super-steps test the delta themselves;
// the host, which reads it after every one in the paper's loop, reads those of
// four at a time.
//
// Triangle counting.  Count(G1, G2, edges) adds, for every edge (u, v), the
// size of the intersection of u's neighbours in G1 and v's neighbours in
// G2.  The paper walks v's slabs in G2 with a warp and lets each lane search
// G1 for (u, w); since an intersection is symmetric, this kernel walks the
// side with fewer buckets (the bucket count grows with the degree) and
// searches the other, which bounds the work of an edge between a hub and a
// leaf by the leaf's degree.
#include "mk_host.h"

#include <algorithm>
#include <cmath>
#include <cstring>
#include <vector>

using namespace mk;

namespace {

constexpr double kFix = 281474976710656.0; // 2^48: fixed-point scale of ranks
constexpr double kInvFix = 1.0 / 281474976710656.0;

// Adds the lanes' values v to *dst with one atomic per warp.
__device__ __forceinline__ void warp_add_u64(unsigned long long *dst, unsigned long long v)
{
    for (int o = 16; o; o >>= 1)
        v += __shfl_xor_sync(kFull, v, o);
    if (lane_id() == 0 && v)
        atomicAdd(dst, v);
}

} // namespace

// ----------------------------------------------------------------- PageRank

namespace {

// Words of a call's counters: rings over the super-steps, so that several go
// out before the host reads anything.  Step i adds the rank without out-edges
// that step i + 1 hands out to dangling[i + 1], its L1 change to delta[i], and
// clears the words of step i + 2.
constexpr uint32_t kRing = 8, kAhead = 4; // steps launched for each read of the deltas
struct PrCtr {
    unsigned long long dangling[kRing], pad[8]; // a line each
    unsigned long long delta[kRing], pad2[8];
    unsigned long long chunks; // of the binned edges
};

// Whether a step before this one met eps: its change is in the ring, and the
// steps after it, which do nothing, leave theirs at zero.  One thread of the
// block reads (a load a warp on that one word took 30 us of a step); *tele
// receives the teleport share of this step.  Called by the whole block.
__device__ __forceinline__ bool pr_done(const PrCtr *ctr, uint32_t step, double eps, uint32_t V = 1,
                                        unsigned long long *tele = nullptr)
{
    __shared__ unsigned long long s_tele;
    bool done = false;
    if (threadIdx.x == 0) {
        done = step && (double)__ldcg(&ctr->delta[(step - 1) % kRing]) * kInvFix <= eps;
        if (tele)
            s_tele = __ldcg(&ctr->dangling[step % kRing]) / V;
    }
    done = __syncthreads_or(done);
    if (tele)
        *tele = s_tele;
    return done;
}

// Adds a and b of every thread to *da and *db, one atomic a block each (one a
// warp made 32,768 of them wait for one word: 57 us a step at 2^20 vertices).
__device__ __forceinline__ void block_add2_u64(unsigned long long *da, unsigned long long a, unsigned long long *db,
                                               unsigned long long b)
{
    __shared__ unsigned long long sa[8], sb[8];
    for (int o = 16; o; o >>= 1) {
        a += __shfl_xor_sync(kFull, a, o);
        b += __shfl_xor_sync(kFull, b, o);
    }
    if (lane_id() == 0) {
        sa[threadIdx.x >> 5] = a;
        sb[threadIdx.x >> 5] = b;
    }
    __syncthreads();
    if (threadIdx.x < 2) {
        unsigned long long t = 0;
        for (int k = 0; k < 8; ++k)
            t += threadIdx.x ? sb[k] : sa[k];
        if (t)
            atomicAdd(threadIdx.x ? db : da, t);
    }
}

// A vertex's out-degree with floor((2^64 - 1) / it), which turns the division
// of a super-step into a multiplication and one correction: for p < 2^63 the
// high product is the quotient or one less.
struct OutDegree {
    unsigned long long inv;
    uint32_t n, pad;
};

// FindContributionPerVertex: contrib[u] = PR[u] / out[u]; the rank of a vertex
// without out-edges is returned for the teleport sum instead.
__device__ __forceinline__ unsigned long long contribution(unsigned long long p, const OutDegree &o,
                                                           unsigned long long *contrib)
{
    unsigned long long q = __umul64hi(p, o.inv);
    q += p - q * o.n >= o.n;
    *contrib = o.n ? q : 0ull;
    return o.n ? 0ull : p;
}

// One block's slabs of a pass over all of them (a contiguous range).
struct SlabRange {
    uint64_t first, last;
};
__device__ __forceinline__ SlabRange block_slabs(const GView &g)
{
    const uint64_t all = (uint64_t)g.H + g.P, per = ((all + gridDim.x - 1) / gridDim.x + 3) & ~3ull;
    const uint64_t a = blockIdx.x * per;
    return {a < all ? a : all, a + per < all ? a + per : all};
}

// The lane's 16 bytes of its slab (eight lanes a slab, four slabs a warp):
// two keys, kEmptyKey where there is none; *own is the slab's owner.
__device__ __forceinline__ void slab_keys(const GView &g, uint64_t s, uint64_t last, uint32_t (&key)[2], uint32_t *own)
{
    const uint32_t part = lane_id() & 7u;
    *own = s < last ? __ldg(&g.owner[s]) : kNil;
    key[0] = key[1] = kEmptyKey;
    if (*own != kNil) { // an unused pool slab holds stale keys
        const uint4 q = __ldcg(reinterpret_cast<const uint4 *>(slab_ptr(g, (uint32_t)s)) + part);
        key[0] = q.x;
        key[1] = part != 7u ? q.z : kEmptyKey;
    }
}

constexpr uint32_t kBinThreads = 1024, kMaxBins = 1024;

} // namespace

// out[u] += live pairs of every slab in use owned by u (one atomic a slab),
// and, with bins, the block's edges into each bin of 2^shift vertices
// (hist[bin * gridDim.x + block]).
template <bool kBins>
__global__ void __launch_bounds__(kBinThreads) k_pr_outdeg(GView g, uint32_t *out, uint32_t shift, uint32_t bins,
                                                           uint32_t *hist)
{
    __shared__ uint32_t h[kMaxBins];
    const uint32_t lane = lane_id(), first = lane & ~7u;
    if (kBins) {
        for (uint32_t i = threadIdx.x; i < bins; i += kBinThreads)
            h[i] = 0;
        __syncthreads();
    }
    const SlabRange r = block_slabs(g);
    for (uint64_t sb = r.first + (threadIdx.x >> 5) * 4; sb < r.last; sb += kBinThreads / 8) {
        uint32_t key[2], own;
        slab_keys(g, sb + (lane >> 3), r.last, key, &own);
        const bool live0 = key[0] < kTombKey, live1 = key[1] < kTombKey;
        const uint32_t n = __popc((__ballot_sync(kFull, live0) >> first) & 0xFFu) +
                           __popc((__ballot_sync(kFull, live1) >> first) & 0xFFu);
        if (lane == first && n)
            atomicAdd(&out[own], n);
        if (kBins) {
            if (live0)
                atomicAdd(&h[key[0] >> shift], 1u);
            if (live1)
                atomicAdd(&h[key[1] >> shift], 1u);
        }
    }
    if (kBins) {
        __syncthreads();
        for (uint32_t i = threadIdx.x; i < bins; i += kBinThreads)
            hist[(uint64_t)i * gridDim.x + blockIdx.x] = h[i];
    }
}

// Writes the block's edges to its places in their destinations' bins, as
// <source, destination> (T = uint2) or, where both fit one word, as the
// source above the destination's place in the bin (T = uint32_t).
template <typename T>
__global__ void __launch_bounds__(kBinThreads) k_pr_bin(GView g, uint32_t shift, uint32_t bins,
                                                        const uint64_t *__restrict__ off, T *edges)
{
    __shared__ uint64_t base[kMaxBins];
    __shared__ uint32_t used[kMaxBins];
    for (uint32_t i = threadIdx.x; i < bins; i += kBinThreads) {
        base[i] = off[(uint64_t)i * gridDim.x + blockIdx.x];
        used[i] = 0;
    }
    __syncthreads();
    const SlabRange r = block_slabs(g);
    for (uint64_t sb = r.first + (threadIdx.x >> 5) * 4; sb < r.last; sb += kBinThreads / 8) {
        uint32_t key[2], own;
        slab_keys(g, sb + (lane_id() >> 3), r.last, key, &own);
#pragma unroll
        for (int k = 0; k < 2; ++k)
            if (key[k] < kTombKey) {
                const uint32_t b = key[k] >> shift;
                T *to = edges + base[b] + atomicAdd(&used[b], 1u);
                if constexpr (sizeof(T) == 8)
                    *to = make_uint2(own, key[k]);
                else
                    *to = own << shift | (key[k] & ((1u << shift) - 1));
            }
    }
}

// The bins in chunks of at most kChunk edges: chunk[i] = <bin, first edge>.
constexpr uint32_t kChunk = 16384;

__global__ void __launch_bounds__(kMaxBins) k_pr_chunks(const uint64_t *__restrict__ off, uint32_t bins,
                                                        uint32_t blocks, ulonglong2 *chunk, PrCtr *ctr)
{
    const uint32_t b = threadIdx.x;
    const uint64_t from = b < bins ? off[(uint64_t)b * blocks] : 0, to = b < bins ? off[(uint64_t)(b + 1) * blocks] : 0;
    const uint64_t n = (to - from + kChunk - 1) / kChunk;
    uint64_t at = n ? atomicAdd(&ctr->chunks, n) : 0;
    for (uint64_t e = from; e < to; e += kChunk)
        chunk[at++] = make_ulonglong2(b, e);
}

// Start vector: 1 / V for every vertex (static), or the caller's ranks
// (incremental / decremental: the ranks before the batch); and what the first
// super-step reads.
__global__ void __launch_bounds__(256) k_pr_start(const float *init, const uint32_t *out, uint32_t V,
                                                  unsigned long long *pr, unsigned long long *contrib,
                                                  unsigned long long *acc, OutDegree *deg, PrCtr *ctr)
{
    unsigned long long dangling = 0;
    for (uint64_t v = blockIdx.x * 256ull + threadIdx.x; v < V; v += gridDim.x * 256ull) {
        const unsigned long long p =
            init ? __double2ull_rn((double)fmaxf(init[v], 0.f) * kFix) : __double2ull_rn(kFix / (double)V);
        pr[v] = p;
        const uint32_t n = out[v];
        deg[v] = {n ? ~0ull / n : 0ull, n, 0u};
        dangling += contribution(p, deg[v], &contrib[v]);
        acc[v] = 0;
    }
    block_add2_u64(&ctr->dangling[0], dangling, &ctr->delta[0], 0ull);
}

// Adds contrib[u] of a chunk's edges u -> v up in shared memory (64-bit sums
// as two words with a carry) and the sums to acc.  A bin's vertices take
// 8 << shift bytes; the edges are read in order and the contributions gathered
// from L2 (8 bytes an edge, 266 G/s at most).  Pushing along the slabs instead
// put one 64-bit atomic an edge on the accumulators in L2, where a power-law
// graph's hubs share a few lines: its slices 50 % busy at most and 13 % on
// average, 339 us a step on R-MAT scale 20 against 48 so, after 310 us
// once a call for the bins.
template <typename T>
__global__ void __launch_bounds__(512) k_pr_pull(const T *__restrict__ edges, const uint64_t *__restrict__ off,
                                                 const ulonglong2 *__restrict__ chunk, uint32_t shift,
                                                 uint32_t blocks, const unsigned long long *__restrict__ contrib,
                                                 unsigned long long *acc, uint32_t V, const PrCtr *ctr, uint32_t step,
                                                 double eps)
{
    extern __shared__ uint32_t sums[]; // low words, then high words
    if (pr_done(ctr, step, eps))
        return;
    const uint32_t width = 1u << shift, mask = width - 1;
    uint32_t *lo = sums, *hi = sums + width;
    const unsigned long long n = __ldg(&ctr->chunks);
    for (unsigned long long c = blockIdx.x; c < n; c += gridDim.x) {
        for (uint32_t i = threadIdx.x; i < 2 * width; i += 512)
            sums[i] = 0;
        const ulonglong2 me = chunk[c];
        const uint64_t end = off[(me.x + 1) * blocks], last = me.y + kChunk < end ? me.y + kChunk : end;
        __syncthreads();
        for (uint64_t i = me.y + threadIdx.x; i < last; i += 4 * 512) {
            uint32_t v[4];
            unsigned long long x[4];
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                const bool in = i + k * 512 < last;
                uint32_t u = kNil;
                v[k] = 0;
                if (in) {
                    const T e = __ldcs(&edges[i + k * 512]);
                    if constexpr (sizeof(T) == 8) {
                        u = e.x;
                        v[k] = e.y & mask;
                    } else {
                        u = e >> shift;
                        v[k] = e & mask;
                    }
                }
                x[k] = in ? __ldg(&contrib[u]) : 0ull;
            }
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                const uint32_t l = (uint32_t)x[k];
                uint32_t h = (uint32_t)(x[k] >> 32);
                if (l)
                    h += atomicAdd(&lo[v[k]], l) + l < l; // the carry
                if (h)
                    atomicAdd(&hi[v[k]], h);
            }
        }
        __syncthreads();
        for (uint32_t i = threadIdx.x; i < width; i += 512) {
            const unsigned long long sum = (unsigned long long)hi[i] << 32 | lo[i];
            if (sum)
                atomicAdd(&acc[(me.x << shift) + i], sum);
        }
        __syncthreads();
    }
}

// Pushes contrib[u] along every live edge u -> v, where the edges are not
// binned.  A warp takes 4 * kPushHalves consecutive slabs a step, four at a
// time: eight lanes a slab, each lane one 16-byte block; the owners, slab
// parts and contributions of every group of four are loaded before any
// atomic, so kPushHalves independent load chains are in flight per lane.
constexpr int kPushHalves = 2;

__global__ void __launch_bounds__(256) k_pr_push(GView g, const unsigned long long *__restrict__ contrib,
                                                 unsigned long long *acc, const PrCtr *ctr, uint32_t step, double eps)
{
    if (pr_done(ctr, step, eps))
        return;
    const uint64_t nslab = (uint64_t)g.H + g.P;
    const uint64_t warp = (blockIdx.x * (uint64_t)blockDim.x + threadIdx.x) >> 5;
    const uint64_t nwarps = ((uint64_t)gridDim.x * blockDim.x) >> 5;
    for (uint64_t s0 = warp * (4 * kPushHalves); s0 < nslab; s0 += nwarps * (4 * kPushHalves)) {
        uint32_t own[kPushHalves], key[kPushHalves][2];
#pragma unroll
        for (int h = 0; h < kPushHalves; ++h)
            slab_keys(g, s0 + h * 4 + (lane_id() >> 3), nslab, key[h], &own[h]);
        unsigned long long c[kPushHalves];
#pragma unroll
        for (int h = 0; h < kPushHalves; ++h)
            c[h] = own[h] != kNil ? __ldg(&contrib[own[h]]) : 0ull;
#pragma unroll
        for (int h = 0; h < kPushHalves; ++h) {
            if (!c[h])
                continue;
            if (key[h][0] < kTombKey)
                atomicAdd(&acc[key[h][0]], c[h]);
            if (key[h][1] < kTombKey)
                atomicAdd(&acc[key[h][1]], c[h]);
        }
    }
}

// Compute + teleport (Eq. 1): PR[v] = (1 - d) / V + d * (acc[v] + teleport
// / V), the L1 delta of the super-step, and what the next one reads.
__global__ void __launch_bounds__(256) k_pr_finish(unsigned long long *pr, unsigned long long *acc,
                                                   const OutDegree *__restrict__ deg, unsigned long long *contrib,
                                                   uint32_t V, double d, unsigned long long base, PrCtr *ctr, uint32_t step, double eps)
{
    unsigned long long tele;
    if (pr_done(ctr, step, eps, V, &tele))
        return;
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        ctr->dangling[(step + 2) % kRing] = 0;
        ctr->delta[(step + 2) % kRing] = 0;
    }
    unsigned long long diff = 0, dangling = 0;
    for (uint64_t v = blockIdx.x * 256ull + threadIdx.x; v < V; v += gridDim.x * 256ull) {
        const unsigned long long nv = base + __double2ull_rn(d * (double)(acc[v] + tele));
        const unsigned long long ov = pr[v];
        diff += nv > ov ? nv - ov : ov - nv;
        pr[v] = nv;
        acc[v] = 0;
        dangling += contribution(nv, deg[v], &contrib[v]);
    }
    block_add2_u64(&ctr->delta[step % kRing], diff, &ctr->dangling[(step + 1) % kRing], dangling);
}

__global__ void k_pr_out(const unsigned long long *pr, uint32_t V, float *out)
{
    const uint32_t v = blockIdx.x * blockDim.x + threadIdx.x;
    if (v < V)
        out[v] = __double2float_rn((double)pr[v] * kInvFix);
}

// ------------------------------------------------------- triangle counting

namespace {

// How many of the warp's n keys (in shared memory) are neighbours of a vertex
// with index entry vi in g: the groups' tally, one count a found key on one
// lane of its group.  Each 4-lane group walks the chain of one key's bucket,
// 32 bytes of a slab a lane, two keys in flight; a lane reading whole slabs by
// itself touched four times as many lines a load (the load pipe 57 % busy).
__device__ __forceinline__ uint32_t count_neighbours(const GView &g, uint2 vi, const uint32_t *keys, uint32_t n,
                                                     uint32_t max_hops)
{
    const uint32_t lane = lane_id(), gi = lane >> 2, s4 = lane & 3u, gbase = lane & ~3u;
    uint32_t count = 0;
    for (uint32_t base = 0; base < n; base += 16) {
        uint32_t key[2], slab[2];
#pragma unroll
        for (uint32_t h = 0; h < 2; ++h) {
            const uint32_t k = base + 8 * h + gi;
            key[h] = k < n ? keys[k] : kNil;
            slab[h] = k < n ? vi.x + bucket_of(key[h], vi.y) : kNil;
        }
        for (uint32_t hop = 0; __any_sync(kFull, slab[0] != kNil || slab[1] != kNil); ++hop) {
            uint4 lo[2], hi[2];
#pragma unroll
            for (uint32_t h = 0; h < 2; ++h) {
                lo[h] = make_uint4(kEmptyKey, 0u, kEmptyKey, 0u);
                hi[h] = make_uint4(kEmptyKey, 0u, kEmptyKey, kNil);
                if (slab[h] != kNil) {
                    const uint4 *p = reinterpret_cast<const uint4 *>(slab_ptr(g, slab[h]) + s4 * 8);
                    lo[h] = __ldcg(p);
                    hi[h] = __ldcg(p + 1);
                }
            }
#pragma unroll
            for (uint32_t h = 0; h < 2; ++h) {
                const bool hit = slab[h] != kNil && (lo[h].x == key[h] || lo[h].z == key[h] || hi[h].x == key[h] ||
                                                     (s4 != 3u && hi[h].z == key[h]));
                count += hit;
                const bool found = (__ballot_sync(kFull, hit) >> gbase) & 0xFu;
                const uint32_t nxt = __shfl_sync(kFull, hi[h].w, gbase + 3);
                slab[h] = found || hop + 1 >= max_hops ? kNil : slab[h] != kNil ? nxt : kNil;
            }
        }
    }
    return count;
}

// |N_g1(u) ∩ N_g2(v)| spread over the warp's lanes (each lane returns its
// share; the full warp calls it with warp-uniform u, v).  The side with
// fewer buckets is walked, eight lists at a time in 4-lane groups (one list,
// slab by slab, by the first group alone), its keys collected in `keys`
// (kTcKeys words of the warp), and looked up in the other side.
constexpr uint32_t kTcKeys = 8 * kPairs;

__device__ __forceinline__ uint32_t warp_edge_count(const GView &g1, const GView &g2, uint32_t u, uint32_t v,
                                                    uint32_t mh1, uint32_t mh2, uint32_t *keys)
{
    const uint32_t lane = lane_id();
    const uint2 vu = __ldg(&g1.vinfo[u]), vv = __ldg(&g2.vinfo[v]);
    // walk N_g2(v) and search g1 for (u, w), or walk N_g1(u) and search g2 for (v, w)
    const bool walk_u = vu.y < vv.y;
    const GView &gw = walk_u ? g1 : g2;
    const GView &gs = walk_u ? g2 : g1;
    const uint2 vw = walk_u ? vu : vv, vs = walk_u ? __ldg(&g2.vinfo[v]) : __ldg(&g1.vinfo[u]);
    const uint32_t mh = walk_u ? mh1 : mh2, mhs = walk_u ? mh2 : mh1;
    const uint32_t g4 = lane >> 2, s4 = lane & 3u, gbase = lane & ~3u;
    uint32_t count = 0;
    for (uint32_t b0 = 0; b0 < vw.y; b0 += 8) {
        uint32_t slab = b0 + g4 < vw.y ? vw.x + b0 + g4 : kNil;
        for (uint32_t hop = 0; __any_sync(kFull, slab != kNil); ++hop) {
            uint4 lo = make_uint4(kEmptyKey, 0u, kEmptyKey, 0u), hi = make_uint4(kEmptyKey, 0u, kEmptyKey, kNil);
            if (slab != kNil) {
                const uint4 *q = reinterpret_cast<const uint4 *>(slab_ptr(gw, slab) + s4 * 8);
                lo = __ldcg(q);
                hi = __ldcg(q + 1);
            }
            const uint32_t key[4] = {lo.x, lo.z, hi.x, s4 == 3u ? kEmptyKey : hi.z};
            uint32_t n = 0;
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                const uint32_t m = __ballot_sync(kFull, key[k] < kTombKey);
                if (key[k] < kTombKey)
                    keys[n + __popc(m & lanemask_lt())] = key[k];
                n += __popc(m);
            }
            __syncwarp();
            count += count_neighbours(gs, vs, keys, n, mhs);
            __syncwarp();
            const uint32_t nxt = __shfl_sync(kFull, hi.w, gbase + 3);
            slab = slab == kNil || hop + 1 >= mh ? kNil : nxt;
        }
    }
    return count;
}

} // namespace

// Count(G1, G2, edges): total += |N_G1(u) ∩ N_G2(v)| over the n edges
// (u, v); a persistent grid whose warps take the edges one at a time from a
// shared counter (*next, zero at launch), so a few edges between two large
// neighbourhoods do not hold up a whole chunk of others.
__global__ void __launch_bounds__(256) k_tc_count(GView g1, GView g2, const uint32_t *__restrict__ src,
                                                  const uint32_t *__restrict__ dst, uint64_t n, uint32_t mh1,
                                                  uint32_t mh2, unsigned long long *total,
                                                  unsigned long long *next)
{
    __shared__ uint32_t keys[8][kTcKeys];
    const uint32_t lane = lane_id();
    unsigned long long count = 0;
    for (;;) {
        unsigned long long e = 0;
        if (lane == 0)
            e = atomicAdd(next, 1ull);
        e = __shfl_sync(kFull, e, 0);
        if (e >= n)
            break;
        const uint32_t u = __ldg(src + e), v = __ldg(dst + e);
        if (u >= g1.V || v >= g2.V) {
            if (lane == 0)
                set_status(g1.st, kErrInvalid);
            continue;
        }
        count += warp_edge_count(g1, g2, u, v, mh1, mh2, keys[threadIdx.x >> 5]);
    }
    warp_add_u64(total, count);
}

namespace {

// Rank of a vertex for the oriented static count: (bucket count, id), a
// strict total order in which vertices with more buckets (higher degree at
// sizing) come later.
__device__ __forceinline__ unsigned long long tc_rank(uint32_t buckets, uint32_t x)
{
    return ((unsigned long long)buckets << 32) | x;
}

// The static count without any copy of the neighbours, for a device that has
// no room for it: a warp takes a slab of u, and for each v there that ranks
// above u looks the keys of u's lists that rank above v up in v's.
__global__ void __launch_bounds__(256) k_tc_walk(GView g, uint32_t max_hops, unsigned long long *total)
{
    __shared__ uint32_t s_keys[8][kPairs + 1];
    const uint32_t lane = lane_id();
    uint32_t *keys = s_keys[threadIdx.x >> 5];
    const uint64_t slabs = (uint64_t)g.H + g.P, nwarps = ((uint64_t)gridDim.x * blockDim.x) >> 5;
    unsigned long long count = 0;
    for (uint64_t c = (blockIdx.x * (uint64_t)blockDim.x + threadIdx.x) >> 5; c < slabs; c += nwarps) {
        const uint32_t u = __ldcg(&g.owner[c]);
        if (u == kNil)
            continue;
        auto above = [&](uint32_t x, unsigned long long rank) {
            return is_key_lane(lane) && x < kTombKey && tc_rank(__ldg(&g.vinfo[x]).y, x) > rank;
        };
        const uint2 vu = __ldg(&g.vinfo[u]);
        const uint32_t x = __ldcg(slab_ptr(g, (uint32_t)c) + lane);
        for (uint32_t todo = __ballot_sync(kFull, above(x, tc_rank(vu.y, u))); todo; todo &= todo - 1) {
            const uint32_t v = __shfl_sync(kFull, x, __ffs(todo) - 1);
            const uint2 vv = __ldg(&g.vinfo[v]);
            for (uint32_t b = 0; b < vu.y; ++b) {
                uint32_t slab = vu.x + b;
                for (uint32_t hop = 0; slab != kNil && hop < max_hops; ++hop) {
                    const uint32_t w = __ldcg(slab_ptr(g, slab) + lane);
                    const bool key = above(w, tc_rank(vv.y, v));
                    const uint32_t m = __ballot_sync(kFull, key);
                    if (key)
                        keys[__popc(m & lanemask_lt())] = w;
                    __syncwarp();
                    if (m)
                        count += count_neighbours(g, vv, keys, __popc(m), max_hops);
                    __syncwarp();
                    slab = __shfl_sync(kFull, w, kNextLane);
                }
            }
        }
    }
    for (int o = 16; o; o >>= 1)
        count += __shfl_xor_sync(kFull, count, o);
    if (lane == 0 && count)
        atomicAdd(total, count);
}

} // namespace

// Static count, each triangle once: with the vertices ranked by tc_rank, a
// triangle a < b < c is counted on its edge (a, b) as the common neighbour c.
// The edges u -> v with rank(u) < rank(v) are first copied out of the slabs
// into one array, vertex by vertex (N+(u)); then, for every u, N+(u) becomes a
// hash set in shared memory, and N+(v) of each v in it is streamed past that
// set: sum over u and v in N+(u) of |N+(u) and N+(v)|.  A test of a streamed
// neighbour moves 4 bytes and looks at one or two words of shared memory; a
// search of v's slab chain for it moved 128 bytes from L2 (R-MAT scale 17,
// 1.9 M undirected edges, 251 M tests: 7.7 ms, 0.6 so).

namespace {

constexpr uint32_t kTcWarp = 32;         // N+(u) of at most this many: one warp, else one block
constexpr uint32_t kTcWarpBits = 8;      // a warp's set: 2^8 words, an eighth full at most
constexpr uint32_t kTcBlockKeys = 1024;  // neighbours of one pass of a block
constexpr uint32_t kTcBlockBits = 13;    // a block's set: up to 2^13 words, an eighth full at most
constexpr uint32_t kTcThreads = 256;

struct TcArrays {
    uint32_t *cnt;             // |N+(u)|
    uint32_t *fill;            // neighbours written so far
    ulonglong2 *list;          // N+(u) at adj[list[u].x], list[u].y of them
    uint32_t *large;           // vertices with more than kTcWarp
    unsigned long long *ctr;   // neighbours in all, vertices in `large`, taken from it, triangles
    uint32_t *adj;
};
enum { kTcTotal = 0, kTcLarge = 1, kTcNext = 2, kTcTriangles = 3, kTcWords = 4 };

__device__ __forceinline__ uint32_t tc_hash(uint32_t x) { return x * 0x9E3779B1u; }

// Enters x in the set of 2^bits words (free words kNil).
__device__ __forceinline__ void tc_enter(uint32_t *set, uint32_t bits, uint32_t x)
{
    uint32_t h = tc_hash(x) >> (32 - bits);
    while (atomicCAS(&set[h], kNil, x) != kNil)
        h = (h + 1) & ((1u << bits) - 1);
}

// Streams N+(v) of the vertices v = row[j], j = first, first + step, ... below
// c, past `lanes` lanes of which the caller is `sub`: test(x) is called with
// the lane's next four neighbours (kNil past a list's end).  A list's place is
// read while the list before it is streamed.
template <typename Test>
__device__ __forceinline__ void tc_stream(const TcArrays &t, const uint32_t *row, uint32_t first, uint32_t c,
                                          uint32_t step, uint32_t sub, uint32_t lanes, Test &&test)
{
    uint32_t j = first;
    ulonglong2 next = j < c ? __ldg(&t.list[row[j]]) : make_ulonglong2(0, 0);
    for (; j < c; j += step) {
        const uint32_t *list = t.adj + next.x;
        const uint32_t n = (uint32_t)next.y;
        if (j + step < c)
            next = __ldg(&t.list[row[j + step]]);
        for (uint32_t i = sub; i < n; i += 4 * lanes) {
            uint32_t x[4];
#pragma unroll
            for (uint32_t k = 0; k < 4; ++k)
                x[k] = i + k * lanes < n ? __ldg(list + i + k * lanes) : kNil;
            test(x);
        }
    }
}

// Bit of vertex x in a bitmap over 2^bits vertices, as <word, bit>: an odd
// multiple modulo 2^bits and a fold, both one to one.  The vertices tested
// most are a power-law graph's hubs, whose ids share most of their bits; by id
// a load of 32 words met 8.8 of them in one bank.
__device__ __forceinline__ uint2 tc_bit(uint32_t x, uint32_t bits)
{
    const uint32_t y = (x * 0x9E3779B1u) & (uint32_t)((1ull << bits) - 1), word = y >> 5;
    return make_uint2(word ^ (word >> 5), y & 31u);
}

// How many of x are in the hash set: four first probes in flight; the few
// that meet another key there go on one by one.
__device__ __forceinline__ uint32_t tc_probe(const uint32_t *set, uint32_t bits, const uint32_t (&x)[4])
{
    const uint32_t mask = (1u << bits) - 1, shift = 32 - bits;
    uint32_t k[4], more = 0, count = 0;
#pragma unroll
    for (uint32_t j = 0; j < 4; ++j)
        k[j] = set[tc_hash(x[j]) >> shift];
#pragma unroll
    for (uint32_t j = 0; j < 4; ++j) {
        count += k[j] == x[j] && x[j] != kNil;
        more |= (k[j] != x[j] && k[j] != kNil && x[j] != kNil ? 1u : 0u) << j;
    }
    while (more) {
        const uint32_t j = __ffs(more) - 1;
        more &= more - 1;
        const uint32_t y = j == 0 ? x[0] : j == 1 ? x[1] : j == 2 ? x[2] : x[3];
        uint32_t h = ((tc_hash(y) >> shift) + 1) & mask, key = set[h];
        while (key != y && key != kNil) {
            h = (h + 1) & mask;
            key = set[h];
        }
        count += key == y;
    }
    return count;
}

} // namespace

// One pass over the slabs in use, eight lanes a slab (16 bytes a lane):
// counts the neighbours that rank above their slab's owner, or (kFill) writes
// them to N+(owner), one atomic a slab.
template <bool kFill>
__global__ void __launch_bounds__(kTcThreads) k_tc_orient(GView g, TcArrays t)
{
    const uint64_t all = (uint64_t)g.H + g.P, stride = ((uint64_t)gridDim.x * kTcThreads) >> 3;
    const uint32_t lane = lane_id(), part = lane & 7u, first = lane & ~7u;
    const uint64_t s0 = (blockIdx.x * (uint64_t)kTcThreads + threadIdx.x) >> 3;
    for (uint64_t sb = s0 & ~3ull; sb < all; sb += stride) { // the warp's four slabs
        const uint64_t s = sb + (lane >> 3);
        const uint32_t u = s < all ? __ldg(&g.owner[s]) : kNil;
        uint4 q = make_uint4(kEmptyKey, 0u, kEmptyKey, 0u);
        unsigned long long ru = ~0ull;
        if (u != kNil) {
            q = __ldcg(reinterpret_cast<const uint4 *>(slab_ptr(g, (uint32_t)s)) + part);
            ru = tc_rank(__ldg(&g.vinfo[u]).y, u);
        }
        const bool up0 = q.x < kTombKey && tc_rank(__ldg(&g.vinfo[q.x]).y, q.x) > ru;
        const bool up1 = part != 7u && q.z < kTombKey && tc_rank(__ldg(&g.vinfo[q.z]).y, q.z) > ru;
        const uint32_t m0 = (__ballot_sync(kFull, up0) >> first) & 0xFFu;
        const uint32_t m1 = (__ballot_sync(kFull, up1) >> first) & 0xFFu;
        const uint32_t n0 = __popc(m0), n = n0 + __popc(m1);
        if (!kFill) {
            if (part == 0 && n)
                atomicAdd(&t.cnt[u], n);
            continue;
        }
        uint32_t base = 0;
        if (part == 0 && n)
            base = atomicAdd(&t.fill[u], n);
        base = __shfl_sync(kFull, base, first);
        if (n) {
            uint32_t *to = t.adj + t.list[u].x + base;
            const uint32_t lt = (1u << part) - 1;
            if (up0)
                to[__popc(m0 & lt)] = q.x;
            if (up1)
                to[n0 + __popc(m1 & lt)] = q.z;
        }
    }
}

// The vertices' places in adj, in blocks of vertices, and the large ones.
__global__ void __launch_bounds__(kTcThreads) k_tc_place(TcArrays t, uint32_t V)
{
    __shared__ uint32_t s_warp[kTcThreads / 32];
    __shared__ unsigned long long s_base;
    const uint32_t v = blockIdx.x * kTcThreads + threadIdx.x, lane = lane_id();
    const uint32_t c = v < V ? t.cnt[v] : 0u;
    uint32_t incl = c;
#pragma unroll
    for (uint32_t o = 1; o < 32; o <<= 1) {
        const uint32_t x = __shfl_up_sync(kFull, incl, o);
        if (lane >= o)
            incl += x;
    }
    if (lane == 31)
        s_warp[threadIdx.x >> 5] = incl;
    __syncthreads();
    if (threadIdx.x == 0) {
        uint32_t sum = 0;
        for (uint32_t k = 0; k < kTcThreads / 32; ++k) {
            const uint32_t x = s_warp[k];
            s_warp[k] = sum;
            sum += x;
        }
        s_base = sum ? atomicAdd(&t.ctr[kTcTotal], (unsigned long long)sum) : 0ull;
    }
    __syncthreads();
    if (v < V)
        t.list[v] = make_ulonglong2(s_base + s_warp[threadIdx.x >> 5] + incl - c, c);
    const uint32_t m = __ballot_sync(kFull, c > kTcWarp);
    unsigned long long base = 0;
    if (m && lane == 0)
        base = atomicAdd(&t.ctr[kTcLarge], (unsigned long long)__popc(m));
    base = __shfl_sync(kFull, base, 0);
    if (c > kTcWarp)
        t.large[base + __popc(m & lanemask_lt())] = v;
}

// Vertices with 2 to kTcWarp neighbours above them, one a warp, four of the
// streamed lists at a time.
__global__ void __launch_bounds__(kTcThreads) k_tc_small(TcArrays t, uint32_t V)
{
    __shared__ uint32_t sets[kTcThreads / 32][1u << kTcWarpBits], rows[kTcThreads / 32][kTcWarp];
    static_assert(8 * kTcWarp <= 1u << kTcWarpBits, "an eighth full");
    const uint32_t lane = lane_id(), w = threadIdx.x >> 5, sub = lane & 7u;
    uint32_t *set = sets[w], *row = rows[w];
    unsigned long long count = 0;
    const uint32_t stride = (gridDim.x * kTcThreads) >> 5;
    for (uint64_t u = (blockIdx.x * kTcThreads + threadIdx.x) >> 5; u < V; u += stride) {
        const ulonglong2 mine = __ldg(&t.list[u]);
        const uint32_t c = (uint32_t)mine.y;
        if (c < 2 || c > kTcWarp)
            continue;
#pragma unroll
        for (uint32_t i = 0; i < 1u << kTcWarpBits; i += 32)
            set[i + lane] = kNil;
        __syncwarp();
        if (lane < c) {
            row[lane] = __ldg(t.adj + mine.x + lane);
            tc_enter(set, kTcWarpBits, row[lane]);
        }
        __syncwarp();
        tc_stream(t, row, lane >> 3, c, 4, sub, 8,
                  [&](const uint32_t(&x)[4]) { count += tc_probe(set, kTcWarpBits, x); });
        __syncwarp();
    }
    warp_add_u64(&t.ctr[kTcTriangles], count);
}

// The vertices with more, one a block at a time (taken from a counter: their
// work differs), the streamed lists one a warp.  With kMap the set is a bitmap
// over all vertices (dynamic shared memory): a test is one load and a shift,
// 10 instructions where the hash set takes 54 and is bound by them (R-MAT
// scale 17: 329 -> 224 us).
template <bool kMap>
__global__ void __launch_bounds__(1024) k_tc_large(TcArrays t, uint32_t vbits)
{
    extern __shared__ uint32_t set[]; // kMap: 2^vbits bits, else 2^kTcBlockBits words
    static_assert(8 * kTcBlockKeys <= 1u << kTcBlockBits, "an eighth full");
    __shared__ unsigned long long s_next;
    const uint32_t lane = lane_id(), w = threadIdx.x >> 5, warps = blockDim.x >> 5;
    const unsigned long long n = t.ctr[kTcLarge];
    unsigned long long count = 0;
    if (kMap)
        for (uint32_t i = threadIdx.x; i < (1u << vbits) / 32; i += blockDim.x)
            set[i] = 0;
    for (;;) {
        __syncthreads();
        if (threadIdx.x == 0)
            s_next = atomicAdd(&t.ctr[kTcNext], 1ull);
        __syncthreads();
        if (s_next >= n)
            break;
        const ulonglong2 list = __ldg(&t.list[t.large[s_next]]);
        const uint32_t c = (uint32_t)list.y, *mine = t.adj + list.x;
        const uint32_t pass = kMap ? c : kTcBlockKeys;
        for (uint32_t at = 0; at < c; at += pass) {
            const uint32_t m = min(c - at, pass);
            const uint32_t bits = 32 - __clz(8 * m - 1);
            if (!kMap) {
                __syncthreads();
                for (uint32_t i = threadIdx.x; i < 1u << bits; i += blockDim.x)
                    set[i] = kNil;
                __syncthreads();
            }
            for (uint32_t i = threadIdx.x; i < m; i += blockDim.x) {
                const uint32_t x = __ldg(mine + at + i);
                const uint2 b = tc_bit(x, vbits);
                if (kMap)
                    atomicOr(&set[b.x], 1u << b.y);
                else
                    tc_enter(set, bits, x);
            }
            __syncthreads();
            uint32_t found = 0;
            tc_stream(t, mine, w, c, warps, lane, 32, [&](const uint32_t(&x)[4]) {
                if (!kMap) {
                    found += tc_probe(set, bits, x);
                    return;
                }
#pragma unroll
                for (int k = 0; k < 4; ++k) {
                    const uint2 at = tc_bit(x[k], vbits);
                    found += x[k] != kNil ? (set[at.x] >> at.y) & 1u : 0u;
                }
            });
            count += found;
            if (kMap) {
                __syncthreads();
                for (uint32_t i = threadIdx.x; i < m; i += blockDim.x)
                    set[tc_bit(__ldg(mine + i), vbits).x] = 0;
            }
        }
    }
    warp_add_u64(&t.ctr[kTcTriangles], count);
}

// ---------------------------------------------------------------- host side

static mk_status tc_walk(mk_graph *g, uint64_t *h_triangles, cudaStream_t s)
{
    unsigned long long *d = nullptr;
    MK_CUDA(pool_alloc((void **)&d, 8, s));
    unsigned long long total = 0;
    mk_status st = cudaMemsetAsync(d, 0, 8, s) == cudaSuccess ? MK_OK : MK_ERR_CUDA;
    if (st == MK_OK)
        st = timed(g, "tc_static", s, 1, [&]() {
            k_tc_walk<<<resident_grid(k_tc_walk, 256), 256, 0, s>>>(g->v, g->v.P + 2, d);
            return cudaSuccess;
        });
    if (st == MK_OK && (cudaMemcpyAsync(&total, d, 8, cudaMemcpyDeviceToHost, s) != cudaSuccess ||
                        cudaStreamSynchronize(s) != cudaSuccess))
        st = MK_ERR_CUDA;
    cudaFreeAsync(d, s);
    *h_triangles = total;
    return st;
}

extern "C" {

mk_status mk_pagerank(mk_graph *g, float *d_pr, int warm_start, float damping, float eps, uint32_t max_iter,
                      uint32_t *h_iters, float *h_delta, void *stream)
{
    if (!g || !d_pr || !(damping > 0.f && damping < 1.f) || !(eps > 0.f) || max_iter == 0)
        return MK_ERR_INVALID_ARG;
    cudaStream_t s = (cudaStream_t)stream;
    const uint32_t V = g->v.V;
    const double d = damping, stop = eps;
    const unsigned long long base = (unsigned long long)std::llround((1.0 - d) / (double)V * kFix);
    mk_status st = MK_OK;
    auto cuda = [&](cudaError_t e) {
        if (st == MK_OK && e != cudaSuccess)
            st = e == cudaErrorMemoryAllocation ? MK_ERR_NO_MEMORY : MK_ERR_CUDA;
        return st == MK_OK;
    };
    // Bins of 2^shift destinations, at most kMaxBins of them: 2^10 vertices
    // (8 KB of sums) up to 2^20 vertices, 2^14 (128 KB) at 2^24.
    uint32_t vbits = 1, shift = 10;
    while (vbits < 32 && (1ull << vbits) < V)
        ++vbits;
    shift = std::max(shift, vbits > 10 ? vbits - 10 : 0u);
    const uint32_t bins = (uint32_t)(((uint64_t)V + (1ull << shift) - 1) >> shift);
    const uint32_t blocks = num_sms() * 2;
    bool binned = shift <= 14 && max_iter >= 4;
    const bool packed = vbits + shift <= 32;
    // per-vertex arrays and counters in one block; the bins' counts and
    // places, and the edges, in another
    unsigned char *vert = nullptr, *bin = nullptr;
    MK_CUDA(pool_alloc((void **)&vert, (size_t)V * (16 + 3 * 8 + 4) + sizeof(PrCtr), s));
    OutDegree *deg = (OutDegree *)vert;
    unsigned long long *pr = (unsigned long long *)(deg + V), *acc = pr + V, *contrib = acc + V;
    PrCtr *ctr = (PrCtr *)(contrib + V);
    uint32_t *out = (uint32_t *)(ctr + 1);
    const uint64_t cells = (uint64_t)bins * blocks + 1;
    const size_t scan_bytes = exclusive_scan_scratch_bytes(cells);
    uint32_t *hist = nullptr;
    uint64_t *off = nullptr, edges_n = 0;
    ulonglong2 *chunk = nullptr;
    void *edges = nullptr;
    cuda(cudaMemsetAsync(ctr, 0, sizeof(PrCtr) + (size_t)V * 4, s));
    if (st == MK_OK && binned) {
        if (pool_alloc((void **)&bin, cells * 12 + 8 + scan_bytes, s) != cudaSuccess) {
            cudaGetLastError();
            bin = nullptr;
            binned = false;
        }
    }
    if (st == MK_OK && binned) {
        off = (uint64_t *)bin;
        void *scratch = off + cells;
        hist = (uint32_t *)((unsigned char *)scratch + scan_bytes);
        int scans = 0;
        cuda(cudaMemsetAsync(hist + cells - 1, 0, 4, s));
        if (st == MK_OK)
            st = timed(g, "pr_outdeg", s, 1, [&]() {
                k_pr_outdeg<true><<<blocks, kBinThreads, 0, s>>>(g->v, out, shift, bins, hist);
                return exclusive_scan_u32_u64(hist, off, cells, scratch, s, &scans);
            });
        g->launches += (uint64_t)scans;
        if (st == MK_OK)
            cuda(cudaMemcpyAsync(g->h_pinned, off + cells - 1, 8, cudaMemcpyDeviceToHost, s));
        if (st == MK_OK && cuda(cudaStreamSynchronize(s))) {
            std::memcpy(&edges_n, g->h_pinned, 8);
            const size_t rec = packed ? 4 : 8, chunks = bins + edges_n / kChunk;
            if (pool_alloc((void **)&chunk, chunks * 16 + edges_n * rec, s) != cudaSuccess) {
                cudaGetLastError();
                chunk = nullptr;
                binned = false;
            } else {
                edges = chunk + chunks;
                st = timed(g, "pr_bin", s, 2, [&]() {
                    k_pr_chunks<<<1, kMaxBins, 0, s>>>(off, bins, blocks, chunk, ctr);
                    if (packed)
                        k_pr_bin<uint32_t><<<blocks, kBinThreads, 0, s>>>(g->v, shift, bins, off, (uint32_t *)edges);
                    else
                        k_pr_bin<uint2><<<blocks, kBinThreads, 0, s>>>(g->v, shift, bins, off, (uint2 *)edges);
                    return cudaSuccess;
                });
            }
        }
    } else if (st == MK_OK) {
        st = timed(g, "pr_outdeg", s, 1, [&]() {
            k_pr_outdeg<false><<<blocks, kBinThreads, 0, s>>>(g->v, out, 0, 0, nullptr);
            return cudaSuccess;
        });
    }
    const uint32_t vgrid = std::min<uint32_t>(grid_for(V, 256), num_sms() * 8);
    if (st == MK_OK)
        st = timed(g, "pr_start", s, 1, [&]() {
            k_pr_start<<<vgrid, 256, 0, s>>>(warm_start ? d_pr : nullptr, out, V, pr, contrib, acc, deg, ctr);
            return cudaSuccess;
        });
    const size_t sums = (size_t)8 << shift;
    const void *pull = packed ? (const void *)k_pr_pull<uint32_t> : (const void *)k_pr_pull<uint2>;
    int per = 1;
    // (the limit for the largest bins, whatever this call's are: the attribute is
    // the function's, and another thread may be about to launch it)
    if (st == MK_OK && binned && cuda(cudaFuncSetAttribute(pull, cudaFuncAttributeMaxDynamicSharedMemorySize, 8 << 14)))
        cuda(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, pull, 512, sums));
    const uint32_t pull_grid = (uint32_t)std::min<uint64_t>((uint64_t)num_sms() * std::max(per, 1), bins + edges_n / kChunk);
    // 4 * kPushHalves slabs per warp step
    const uint32_t push_grid = std::min<uint64_t>(grid_for(((uint64_t)g->v.H + g->v.P) * 32 / (4 * kPushHalves), 256),
                                                  (uint64_t)resident_grid(k_pr_push, 256) * 4);
    uint32_t it = 0;
    double delta = 0;
    for (bool met = false; st == MK_OK && !met && it < max_iter;) {
        const uint32_t n = std::min(kAhead, max_iter - it);
        for (uint32_t k = 0; k < n && st == MK_OK; ++k) {
            uint32_t step = it + k;
            st = timed(g, "pr_step", s, 2, [&]() {
                if (binned) {
                    void *args[] = {&edges, &off, &chunk, &shift, (void *)&blocks, &contrib, &acc, (void *)&V, &ctr,
                                    &step, (void *)&stop};
                    const cudaError_t e = cudaLaunchKernel(pull, dim3(pull_grid), dim3(512), args, sums, s);
                    if (e != cudaSuccess)
                        return e;
                } else {
                    k_pr_push<<<push_grid, 256, 0, s>>>(g->v, contrib, acc, ctr, step, stop);
                }
                k_pr_finish<<<vgrid, 256, 0, s>>>(pr, acc, deg, contrib, V, d, base, ctr, step, stop);
                return cudaSuccess;
            });
        }
        if (st == MK_OK)
            cuda(cudaMemcpyAsync(g->h_pinned, ctr->delta, sizeof ctr->delta, cudaMemcpyDeviceToHost, s));
        if (st == MK_OK)
            cuda(cudaStreamSynchronize(s));
        for (uint32_t k = 0; k < n && st == MK_OK && !met; ++k, ++it) {
            unsigned long long dfx = 0;
            std::memcpy(&dfx, g->h_pinned + 2 * (it % kRing), 8);
            delta = (double)dfx * kInvFix;
            met = delta <= stop;
        }
    }
    if (st == MK_OK)
        st = timed(g, "pr_out", s, 1, [&]() {
            k_pr_out<<<grid_for(V, 256), 256, 0, s>>>(pr, V, d_pr);
            return cudaSuccess;
        });
    cudaFreeAsync(vert, s);
    if (bin)
        cudaFreeAsync(bin, s);
    if (chunk)
        cudaFreeAsync(chunk, s);
    if (h_iters)
        *h_iters = it;
    if (h_delta)
        *h_delta = (float)delta;
    return st;
}

mk_status mk_tc_count(mk_graph *g1, mk_graph *g2, const uint32_t *d_src, const uint32_t *d_dst, uint64_t n,
                      unsigned long long *d_total, void *stream)
{
    if (!g1 || !g2 || !d_total || (n && (!d_src || !d_dst)) || g1->v.V != g2->v.V)
        return MK_ERR_INVALID_ARG;
    if (!n)
        return MK_OK;
    cudaStream_t s = (cudaStream_t)stream;
    const uint32_t grid = std::min<uint64_t>(grid_for(n * 32, 256), (uint64_t)resident_grid(k_tc_count, 256));
    unsigned long long *next = nullptr;
    MK_CUDA(pool_alloc((void **)&next, 8, s));
    MK_CUDA(cudaMemsetAsync(next, 0, 8, s));
    const mk_status st = timed(g1, "tc_count", s, 1, [&]() {
        k_tc_count<<<grid, 256, 0, s>>>(g1->v, g2->v, d_src, d_dst, n, g1->v.P + 2, g2->v.P + 2, d_total, next);
        return cudaSuccess;
    });
    cudaFreeAsync(next, s);
    return st;
}

mk_status mk_tc_static(mk_graph *g, uint64_t *h_triangles, void *stream)
{
    if (!g || !h_triangles)
        return MK_ERR_INVALID_ARG;
    cudaStream_t s = (cudaStream_t)stream;
    const uint64_t V = g->v.V;
    // the per-vertex arrays in one block, the neighbours (as many as there
    // are, read back first) in another
    unsigned char *block = nullptr;
    const size_t bytes = V * (16 + 4 + 4 + 4) + kTcWords * 8;
    if (g->dbg_no_scratch || pool_alloc((void **)&block, bytes, s) != cudaSuccess)
        return tc_walk(g, h_triangles, s);
    TcArrays t{};
    t.list = (ulonglong2 *)block;
    t.ctr = (unsigned long long *)(t.list + V);
    t.cnt = (uint32_t *)(t.ctr + kTcWords);
    t.fill = t.cnt + V;
    t.large = t.fill + V;
    const uint32_t slab_grid = resident_grid(k_tc_orient<false>, kTcThreads);
    unsigned long long total = 0;
    mk_status st = MK_OK;
    auto cuda = [&](cudaError_t e) {
        if (st == MK_OK && e != cudaSuccess)
            st = e == cudaErrorMemoryAllocation ? MK_ERR_NO_MEMORY : MK_ERR_CUDA;
        return st == MK_OK;
    };
    if (cuda(cudaMemsetAsync(t.ctr, 0, kTcWords * 8 + V * 8, s)))
        st = timed(g, "tc_orient", s, 2, [&]() {
            k_tc_orient<false><<<slab_grid, kTcThreads, 0, s>>>(g->v, t);
            k_tc_place<<<grid_for(V, kTcThreads), kTcThreads, 0, s>>>(t, (uint32_t)V);
            return cudaSuccess;
        });
    if (st == MK_OK)
        cuda(cudaMemcpyAsync(&total, t.ctr + kTcTotal, 8, cudaMemcpyDeviceToHost, s));
    if (st == MK_OK)
        cuda(cudaStreamSynchronize(s));
    if (st == MK_OK && total) {
        if (pool_alloc((void **)&t.adj, total * 4, s) != cudaSuccess) {
            cudaFreeAsync(block, s);
            return tc_walk(g, h_triangles, s);
        }
        if (st == MK_OK)
            st = timed(g, "tc_static", s, 3, [&]() {
                k_tc_orient<true><<<slab_grid, kTcThreads, 0, s>>>(g->v, t);
                // a bitmap of up to 128 KB (2^20 vertices), with blocks large
                // enough that those an SM holds fill it
                uint32_t vbits = 5;
                while (vbits < 32 && (1ull << vbits) < V)
                    ++vbits;
                const size_t map = (1ull << vbits) / 8;
                constexpr size_t kMapMax = 128u << 10, kSets = sizeof(uint32_t) << kTcBlockBits;
                const bool use_map = map <= kMapMax;
                const size_t smem = use_map ? map : kSets;
                const int threads = smem <= 24u << 10 ? 256 : smem <= 48u << 10 ? 512 : 1024;
                const void *k = use_map ? (const void *)k_tc_large<true> : (const void *)k_tc_large<false>;
                int per = 0;
                // (not `smem`: another thread may be about to launch the same kernel)
                cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                                     (int)(use_map ? kMapMax : kSets));
                if (e == cudaSuccess)
                    e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, k, threads, smem);
                if (e != cudaSuccess)
                    return e;
                void *args[] = {&t, &vbits};
                e = cudaLaunchKernel(k, dim3(num_sms() * std::max(per, 1)), dim3(threads), args, smem, s);
                if (e != cudaSuccess)
                    return e;
                k_tc_small<<<resident_grid(k_tc_small, kTcThreads), kTcThreads, 0, s>>>(t, (uint32_t)V);
                return cudaSuccess;
            });
        total = 0;
        if (st == MK_OK)
            cuda(cudaMemcpyAsync(&total, t.ctr + kTcTriangles, 8, cudaMemcpyDeviceToHost, s));
        if (st == MK_OK)
            cuda(cudaStreamSynchronize(s));
        if (t.adj)
            cudaFreeAsync(t.adj, s);
    }
    cudaFreeAsync(block, s);
    *h_triangles = total;
    return st;
}

mk_status mk_tc_update(mk_graph *g_post, mk_graph *g_upd, const uint32_t *d_src, const uint32_t *d_dst, uint64_t n,
                       int deletion, int64_t *h_delta, void *stream)
{
    if (!g_post || !g_upd || !h_delta || g_post->v.V != g_upd->v.V || (n && (!d_src || !d_dst)))
        return MK_ERR_INVALID_ARG;
    cudaStream_t s = (cudaStream_t)stream;
    unsigned long long *d = nullptr;
    MK_CUDA(pool_alloc((void **)&d, 24, s));
    MK_CUDA(cudaMemsetAsync(d, 0, 24, s));
    mk_status st = mk_tc_count(g_post, g_post, d_src, d_dst, n, d + 0, stream);
    if (st == MK_OK)
        st = mk_tc_count(g_post, g_upd, d_src, d_dst, n, d + 1, stream);
    if (st == MK_OK)
        st = mk_tc_count(g_upd, g_upd, d_src, d_dst, n, d + 2, stream);
    unsigned long long S[3] = {0, 0, 0};
    if (st == MK_OK && (cudaMemcpyAsync(S, d, 24, cudaMemcpyDeviceToHost, s) != cudaSuccess ||
                        cudaStreamSynchronize(s) != cudaSuccess))
        st = MK_ERR_CUDA;
    cudaFreeAsync(d, s);
    if (st != MK_OK)
        return st;
    // S1 = 2 T1 + 4 T2 + 6 T3 and S2 = 2 T2 + 6 T3 (insertion) or S1 = 2 T1,
    // S2 = 2 T2 (deletion); S3 = 6 T3 in both
    const long long s1 = (long long)S[0], s2 = (long long)S[1], s3 = (long long)S[2];
    if (s1 % 2 || s2 % 2 || s3 % 6)
        return MK_ERR_INTERNAL;
    *h_delta = deletion ? -(s1 / 2 + s2 / 2 + s3 / 6) : (s1 / 2 - s2 / 2 + s3 / 6);
    return MK_OK;
}

} // extern "C"
