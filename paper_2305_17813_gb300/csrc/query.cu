// Batched edge query (paper, Sec. "Experimental Evaluation", query: the
// destination is hashed to one bucket of the source and only that chain is
// walked; the walk stops at the key or at the chain's end).
//
// Queries are independent, so the batch is not sorted.  One warp answers 32
// consecutive queries (a chunk): each lane fetches the source's bucket range
// for its own query, then the warp reads the 32 head slabs at once, G lanes a
// slab, each lane 32/G consecutive words of the 128 bytes as one vector (G =
// 8: 16 bytes, two pairs per lane; G = 32: one word per lane, the paper's
// layout) - 32 registers a lane whatever G is - and examines them; chains
// that go on are read in further rounds of the same kind.  A lookup is one
// slab of DRAM out of order, so what bounds a large batch is how many slabs
// are in flight.  R-MAT scale 20, 2.1 M lookups, half of them present: 74 us
// with 32/G chains in flight a warp, 54 us so (the slabs alone, as one random
// gather of 128-byte lines: 33-45 us).  The warp writes one bitmap word per
// chunk.  G and the block size are picked by the autotuner
// (mk_autotune); the default is G = 8, 256 threads.
//
// The multi-request form runs the chunks of many query requests in one
// persistent grid-stride launch: chunk c belongs to the request whose chunk
// range [prefix[r], prefix[r+1]) contains it, so uneven requests share one
// launch (and one CUDA graph node) instead of one launch each.
#include "mk_host.h"
#include "mk_query.h"

#include <algorithm>
#include <cstring>
#include <type_traits>

using namespace mk;

namespace {

template <int W>
struct Vec;
template <>
struct Vec<1> {
    static __device__ __forceinline__ void load(const uint32_t *p, uint32_t *w) { w[0] = __ldg(p); }
};
template <>
struct Vec<2> {
    static __device__ __forceinline__ void load(const uint32_t *p, uint32_t *w)
    {
        const uint2 x = __ldg(reinterpret_cast<const uint2 *>(p));
        w[0] = x.x;
        w[1] = x.y;
    }
};
template <>
struct Vec<4> {
    static __device__ __forceinline__ void load(const uint32_t *p, uint32_t *w)
    {
        const uint4 x = __ldg(reinterpret_cast<const uint4 *>(p));
        w[0] = x.x;
        w[1] = x.y;
        w[2] = x.z;
        w[3] = x.w;
    }
};
template <>
struct Vec<8> {
    static __device__ __forceinline__ void load(const uint32_t *p, uint32_t *w)
    {
        Vec<4>::load(p, w);
        Vec<4>::load(p + 4, w + 4);
    }
};

// A lane's query: its destination and its source's buckets; none (vi.y 0, and
// kNil, which no key word holds) where there is no query or a rejected one.
struct Lookup {
    uint32_t d;
    uint2 vi;
};

__device__ __forceinline__ Lookup look_up(const GView &g, uint32_t s, uint32_t d, bool live)
{
    Lookup q{kNil, make_uint2(0u, 0u)};
    const bool bad = live && (s >= g.V || d >= g.V);
    if (live && !bad)
        q = {d, __ldg(&g.vinfo[s])};
    if (__any_sync(kFull, bad) && lane_id() == 0)
        set_status(g.st, kErrInvalid);
    return q;
}

// Answers the warp's 32 queries (a lane's own if `live`) of one request.  A
// round reads and examines a slab of every query left.  A lane that finds the
// key notes the pair's number in four bits of its own for each slab it reads;
// the G lanes of a group put theirs together at the end of the round, where
// the query's own lane takes its four bits and reads one more word of the
// slab (in L1 by now): the weight, or the link of a chain that goes on.  290
// instructions a chunk; a form that votes on hits and on free pairs at each
// step and picks the weight out of registers took 600.  (A chain need not end
// at a free pair: its slabs fill up in order, so the next link is null there.)
template <int G>
__device__ __forceinline__ void query_chunk(const GView &g, const Lookup &q, bool live,
                                            uint32_t *__restrict__ bitmap_word, uint32_t *__restrict__ w_out,
                                            uint32_t max_hops, uint32_t &loads)
{
    constexpr uint32_t W = 32 / G;        // words per lane
    constexpr uint32_t kGroups = 32 / G;  // slabs a warp-wide load reads
    constexpr uint32_t kSteps = 32 / kGroups;
    constexpr uint32_t kAcc = (kSteps + 7) / 8; // words of notes, eight steps each
    const uint32_t lane = lane_id(), gi = lane / G, sub = lane % G;
    // numbers of this lane's pairs, from 1; zero where a word is no key
    uint32_t code[(W + 1) / 2];
#pragma unroll
    for (uint32_t j = 0; j < W; j += 2)
        code[j / 2] = is_key_lane(sub * W + j) ? (sub * W + j) / 2 + 1 : 0u;
    uint32_t slab = q.vi.y ? q.vi.x + bucket_of(q.d, q.vi.y) : kNil, wt = 0;
    bool found = false;
    uint32_t act = __ballot_sync(kFull, slab != kNil);
    auto round = [&](auto all) {
        constexpr bool kAll = decltype(all)::value;
        auto skip = [&](uint32_t k) { return !kAll && ((act >> (k * kGroups)) & ((1u << kGroups) - 1u)) == 0; };
        uint32_t w[kSteps][W], note[kAcc];
#pragma unroll
        for (uint32_t k = 0; k < kSteps; ++k) {
            // a query that is answered, or none, reads slab 0 along with the others of its step
            const uint32_t at = __shfl_sync(kFull, slab, k * kGroups + gi);
            if (!skip(k))
                Vec<W>::load(slab_ptr(g, at != kNil ? at : 0u) + sub * W, w[k]);
        }
#pragma unroll
        for (uint32_t i = 0; i < kAcc; ++i)
            note[i] = 0;
#pragma unroll
        for (uint32_t k = 0; k < kSteps; ++k) {
            if (skip(k))
                continue;
            const uint32_t d = __shfl_sync(kFull, q.d, k * kGroups + gi);
#pragma unroll
            for (uint32_t j = 0; j < W; j += 2)
                // At most one pair adds to a step's four bits: a list holds a
                // vertex once, and d is a vertex or kNil.  (The key of a free
                // or deleted pair as d would match many, and their sum carry
                // into the bits of another query.)
                if (w[k][j] == d)
                    note[k / 8] += code[j / 2] << (4 * (k % 8));
        }
        uint32_t mine = 0;
#pragma unroll
        for (uint32_t i = 0; i < kAcc; ++i) {
#pragma unroll
            for (uint32_t o = 1; o < G; o <<= 1)
                note[i] |= __shfl_xor_sync(kFull, note[i], o);
            const uint32_t v = __shfl_sync(kFull, note[i], (lane % kGroups) * G);
            mine = lane / kGroups / 8 == i ? v : mine;
        }
        const uint32_t pos = (mine >> (4 * ((lane / kGroups) % 8))) & 15u;
        if (slab != kNil) {
            const uint32_t word = __ldg(slab_ptr(g, slab) + (pos ? 2 * pos - 1 : 31u));
            found = pos != 0;
            wt = found ? word : 0u;
            slab = found ? kNil : word;
        }
    };
    if (act) {
        loads += __popc(act);
        round(std::true_type{});
        act = __ballot_sync(kFull, slab != kNil);
        for (uint32_t hop = 0; act && hop < max_hops; ++hop) {
            loads += __popc(act);
            round(std::false_type{});
            act = __ballot_sync(kFull, slab != kNil);
        }
    }
    const uint32_t bits = __ballot_sync(kFull, found);
    if (w_out && live)
        w_out[lane] = wt;
    if (lane == 0)
        *bitmap_word = bits;
}

// Warps stride over the chunks; the queries of the chunk after next and the
// bucket range of the next are in flight while a chunk is answered (82 us where
// the head slabs were worked out as soon as the bucket ranges were asked for).
template <int G>
__global__ void __launch_bounds__(512, kQueryThreads / 512)
k_query(GView g, const uint32_t *__restrict__ src, const uint32_t *__restrict__ dst, uint32_t n,
        uint32_t *__restrict__ bitmap, uint32_t *__restrict__ w_out, uint32_t max_hops)
{
    const uint32_t stride = gridDim.x * blockDim.x; // queries, a lane's next is this far
    uint64_t i = blockIdx.x * blockDim.x + threadIdx.x;
    if ((i & ~31ull) >= n || status_hint(g.st) != 0)
        return;
    uint32_t s1 = 0, d1 = 0, loads = 0;
    auto fetch = [&](uint64_t at) {
        if (at < n) {
            s1 = __ldg(src + at);
            d1 = __ldg(dst + at);
        }
    };
    fetch(i);
    Lookup q = look_up(g, s1, d1, i < n);
    fetch(i + stride);
    for (; (i & ~31ull) < n; i += stride) {
        const Lookup next = look_up(g, s1, d1, i + stride < n);
        fetch(i + 2ull * stride);
        query_chunk<G>(g, q, i < n, bitmap + i / 32, w_out ? w_out + (i & ~31ull) : nullptr, max_hops, loads);
        q = next;
    }
    count_add(g.st, kCtrQuerySlabs, loads);
}

template <int G>
__global__ void __launch_bounds__(512, kQueryThreads / 512)
k_query_multi(GView g, const QueryReq *__restrict__ reqs, const uint64_t *__restrict__ prefix, uint32_t nreq_max,
              const uint64_t *__restrict__ total, uint32_t max_hops)
{
    if (status_hint(g.st) != 0)
        return;
    const uint64_t nchunks = total[0];
    const uint32_t nreq = total[1] < nreq_max ? (uint32_t)total[1] : nreq_max;
    const uint64_t warp0 = (blockIdx.x * (uint64_t)blockDim.x + threadIdx.x) >> 5;
    const uint64_t nwarps = ((uint64_t)gridDim.x * blockDim.x) >> 5;
    uint32_t loads = 0;
    for (uint64_t c = warp0; c < nchunks; c += nwarps) {
        // request r with prefix[r] <= c < prefix[r + 1]
        uint32_t lo = 0, hi = nreq;
        while (hi - lo > 1) {
            const uint32_t mid = (lo + hi) >> 1;
            if (prefix[mid] <= c)
                lo = mid;
            else
                hi = mid;
        }
        const QueryReq r = reqs[lo];
        const uint64_t local = c - prefix[lo], at = local * 32 + lane_id();
        const bool live = at < r.n;
        const Lookup q = look_up(g, live ? __ldg(r.src + at) : 0u, live ? __ldg(r.dst + at) : 0u, live);
        query_chunk<G>(g, q, live, r.bitmap + local, r.w ? r.w + local * 32 : nullptr, max_hops, loads);
    }
    count_add(g.st, kCtrQuerySlabs, loads);
}

} // namespace

namespace mk {

cudaError_t launch_query(mk_graph *g, int group, int block, const uint32_t *src, const uint32_t *dst, uint64_t n,
                         uint32_t *bitmap, uint32_t *w, cudaStream_t s)
{
    const uint32_t max_hops = g->v.P + 2;
    auto go = [&](auto kernel) {
        const uint32_t grid = std::min(grid_for(n, (uint32_t)block), (uint32_t)num_sms() * (kQueryThreads / block));
        kernel<<<grid, block, 0, s>>>(g->v, src, dst, (uint32_t)n, bitmap, w, max_hops);
    };
    switch (group) {
    case 4: go(k_query<4>); break;
    case 16: go(k_query<16>); break;
    case 32: go(k_query<32>); break;
    default: go(k_query<8>); break;
    }
    return cudaGetLastError();
}

cudaError_t launch_query_multi(mk_graph *g, int group, int block, int grid, const QueryReq *reqs,
                               const uint64_t *prefix, uint32_t nreq, const uint64_t *total, cudaStream_t s)
{
    const uint32_t max_hops = g->v.P + 2;
    switch (group) {
    case 4: k_query_multi<4><<<grid, block, 0, s>>>(g->v, reqs, prefix, nreq, total, max_hops); break;
    case 16: k_query_multi<16><<<grid, block, 0, s>>>(g->v, reqs, prefix, nreq, total, max_hops); break;
    case 32: k_query_multi<32><<<grid, block, 0, s>>>(g->v, reqs, prefix, nreq, total, max_hops); break;
    default: k_query_multi<8><<<grid, block, 0, s>>>(g->v, reqs, prefix, nreq, total, max_hops); break;
    }
    return cudaGetLastError();
}

} // namespace mk

extern "C" mk_status mk_query_batch(mk_graph *g, const uint32_t *d_src, const uint32_t *d_dst, uint64_t n,
                                    uint32_t *d_bitmap, uint32_t *d_w, void *stream)
{
    if (!g || (n > 0 && (!d_src || !d_dst || !d_bitmap)) || n >= 0xFFFFFFFFull)
        return MK_ERR_INVALID_ARG;
    cudaStream_t s = (cudaStream_t)stream;
    if (n == 0)
        return MK_OK;
    return timed(g, "query", s, 1, [&]() {
        return launch_query(g, g->tune.query_group, g->tune.query_block, d_src, d_dst, n, d_bitmap, d_w, s);
    });
}
