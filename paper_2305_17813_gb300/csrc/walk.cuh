// Slab-list traversal and frontier helpers shared by the algorithm kernels.
#pragma once

#include "mk_device.cuh"

namespace mk {

// A block's staging area for frontier entries: a buffer a warp, so that
// nothing is shared while a round runs.  A full buffer goes to the global
// frontier with one atomicAdd on its count (at least kWarpBuf / 2 entries at
// a time); what is left at the end of a round with one a block
// (frontier_flush).  Thousands of warps meet on that one count: with one
// buffer a block, and an atomic for every later append of a warp, the static
// BFS on R-MAT scale 20 waited for the count most of the time.
constexpr uint32_t kWarpBuf = 64;
template <uint32_t kWarps>
struct FrontierSmem {
    uint2 buf[kWarps][kWarpBuf];
    uint32_t held[kWarps]; // entries in each warp's buffer
    uint32_t at[kWarps];   // their places at a flush
};

template <uint32_t kWarps>
__device__ __forceinline__ void frontier_init(FrontierSmem<kWarps> &sm)
{
    if (threadIdx.x < kWarps)
        sm.held[threadIdx.x] = 0;
    __syncthreads();
}

// Appends the slab lists of the lane's vertices y[k] with up[k] (vi[k]: its
// vinfo entry) to the frontier as <list, y> entries (the source travels with
// the list, so a consumer needs no list_src lookup): one scan over the warp
// and at most one reservation for all of them (one for each vertex with many
// buckets made the round after a hub wait for 25 of them in a row).  Must be
// called by the full warp; sets
// *overflow for an entry that would not fit in `cap`.  The count is a 32-bit
// word, or the low half of a 64-bit one: every access to a word that blocks
// race on has the word's own width.
template <int N, uint32_t kWarps, typename C>
__device__ __forceinline__ void enqueue_lists(FrontierSmem<kWarps> &sm, const uint32_t (&y)[N], const bool (&up)[N],
                                              const uint2 (&vi)[N], uint2 *out, C *count, uint32_t cap,
                                              int *overflow)
{
    constexpr uint32_t kSmall = 8;
    const uint32_t lane = lane_id(), w = threadIdx.x >> 5;
    uint32_t c = 0;
    bool big = false;
#pragma unroll
    for (int k = 0; k < N; ++k) {
        c += up[k] ? vi[k].y : 0u;
        big = big || (up[k] && vi[k].y > kSmall);
    }
    if (!__any_sync(kFull, c != 0))
        return;
    uint32_t incl = c;
#pragma unroll
    for (uint32_t o = 1; o < 32; o <<= 1) {
        const uint32_t t = __shfl_up_sync(kFull, incl, o);
        if (lane >= o)
            incl += t;
    }
    const uint32_t total = __shfl_sync(kFull, incl, 31), held = sm.held[w];
    const bool any_big = __any_sync(kFull, big), fits = !any_big && held + total <= kWarpBuf;
    auto put = [&](uint32_t at, uint2 ent) {
        if (at < cap)
            out[at] = ent;
        else
            *overflow = 1;
    };
    uint32_t base = 0;
    if (!fits) {
        if (lane == 0)
            base = (uint32_t)atomicAdd(count, (C)(held + total));
        base = __shfl_sync(kFull, base, 0);
        for (uint32_t t = lane; t < held; t += 32)
            put(base + t, sm.buf[w][t]);
    }
    uint32_t t = held + incl - c;
#pragma unroll
    for (int k = 0; k < N; ++k) {
        const uint32_t nb = up[k] ? vi[k].y : 0u;
        if (nb <= kSmall)
            for (uint32_t b = 0; b < nb; ++b) {
                if (fits)
                    sm.buf[w][t + b] = make_uint2(vi[k].x + b, y[k]);
                else
                    put(base + t + b, make_uint2(vi[k].x + b, y[k]));
            }
        if (any_big)
            for (uint32_t m = __ballot_sync(kFull, nb > kSmall); m; m &= m - 1) {
                const uint32_t l = __ffs(m) - 1;
                const uint32_t first = __shfl_sync(kFull, vi[k].x, l), n = __shfl_sync(kFull, nb, l);
                const uint32_t yl = __shfl_sync(kFull, y[k], l), at = base + __shfl_sync(kFull, t, l);
                for (uint32_t b = lane; b < n; b += 32)
                    put(at + b, make_uint2(first + b, yl));
            }
        t += nb;
    }
    __syncwarp();
    if (lane == 0)
        sm.held[w] = fits ? held + total : 0u;
    __syncwarp();
}

// Copies the block's staged entries to the global frontier and empties the
// staging area.  Called by every thread of the block; the caller synchronises
// the block before the entries or the staging area are used again.  `beside`
// is called by the block's second warp while the first one waits for its
// places: another reservation of the round.
template <uint32_t kWarps, typename C, typename F>
__device__ __forceinline__ void frontier_flush(FrontierSmem<kWarps> &sm, uint2 *out, C *count, uint32_t cap,
                                               int *overflow, F &&beside)
{
    const uint32_t lane = lane_id(), w = threadIdx.x >> 5;
    __syncthreads();
    if (w == 0) {
        const uint32_t h = lane < kWarps ? sm.held[lane] : 0u;
        uint32_t incl = h;
#pragma unroll
        for (uint32_t o = 1; o < 32; o <<= 1) {
            const uint32_t t = __shfl_up_sync(kFull, incl, o);
            if (lane >= o)
                incl += t;
        }
        uint32_t base = 0;
        if (lane == 31 && incl)
            base = (uint32_t)atomicAdd(count, (C)incl);
        base = __shfl_sync(kFull, base, 31);
        if (lane < kWarps)
            sm.at[lane] = base + incl - h;
    } else if (w == 1) {
        beside();
    }
    __syncthreads();
    const uint32_t held = sm.held[w], at = sm.at[w];
    for (uint32_t t = lane; t < held; t += 32) {
        if (at + t < cap)
            out[at + t] = sm.buf[w][t];
        else
            *overflow = 1;
    }
    __syncwarp();
    if (lane == 0)
        sm.held[w] = 0;
}

template <uint32_t kWarps, typename C>
__device__ __forceinline__ void frontier_flush(FrontierSmem<kWarps> &sm, uint2 *out, C *count, uint32_t cap,
                                               int *overflow)
{
    frontier_flush(sm, out, count, cap, overflow, []() {});
}

} // namespace mk

namespace mk {

// Tiled walk: each 4-lane group of the warp walks its own slab list (eight
// lists per warp, so a warp has eight slab loads in flight instead of one);
// lane s4 of a group holds words 8*s4 .. 8*s4+7 of the slab as two 16-byte
// vectors, i.e. pairs 4*s4 .. 4*s4+3 (lane 3: pairs 12-14, then the unused
// lane and the next lane).  `slab` and `first_lane` are per group (kNil =
// the group has no list).  Per slab, f(key, weight, live) is called once by
// every lane of the warp (convergent) with the lane's four pairs as arrays
// (key[k], weight[k], live[k], k = 0..3), so that the callee can put the
// memory accesses of all four in flight together; `live` is false for free /
// deleted keys, for key words below first_lane on the first slab, and for
// groups without a list.  With have_first, (lo0, hi0) already hold the
// lane's part of `slab` (group4_load), loaded ahead by the caller.  Stops
// after the slab whose next lane is null or after max_hops slabs; returns
// the number of slabs loaded by the warp.
template <typename F>
__device__ __forceinline__ uint32_t walk_lists_g4_from(const GView &g, uint32_t slab, bool have_first, uint4 lo0,
                                                       uint4 hi0, uint32_t first_lane, uint32_t max_hops, F &&f)
{
    const uint32_t lane = lane_id(), s4 = lane & 3u, gbase = lane & ~3u;
    bool active = slab != kNil;
    uint32_t loads = 0;
    for (uint32_t hop = 0; __any_sync(kFull, active); ++hop) {
        uint4 lo = make_uint4(kEmptyKey, kFull, kFull, kFull), hi = lo;
        if (hop == 0 && have_first) {
            lo = lo0;
            hi = hi0;
        } else if (active) {
            const uint4 *p = reinterpret_cast<const uint4 *>(slab_ptr(g, slab) + s4 * 8);
            lo = __ldcg(p);
            hi = __ldcg(p + 1);
        }
        loads += __popc(__ballot_sync(kFull, active && s4 == 0));
        const uint32_t w0 = 8 * s4;
        const uint32_t key[4] = {lo.x, lo.z, hi.x, hi.z}, wt[4] = {lo.y, lo.w, hi.y, hi.w};
        const bool live[4] = {active && lo.x < kTombKey && w0 >= first_lane,
                              active && lo.z < kTombKey && w0 + 2 >= first_lane,
                              active && hi.x < kTombKey && w0 + 4 >= first_lane,
                              active && s4 != 3u && hi.z < kTombKey && w0 + 6 >= first_lane};
        f(key, wt, live);
        const uint32_t nxt = __shfl_sync(kFull, hi.w, gbase + 3);
        if (active) {
            if (nxt == kNil || hop + 1 >= max_hops)
                active = false;
            else
                slab = nxt;
        }
        first_lane = 0;
    }
    return loads;
}

// The lane's 32-byte part of slab s for a 4-lane group (words 8*s4 ..
// 8*s4+7); empty parts for s == kNil.
__device__ __forceinline__ void group4_load(const GView &g, uint32_t s, uint4 &lo, uint4 &hi)
{
    lo = make_uint4(kEmptyKey, kFull, kFull, kFull);
    hi = lo;
    if (s != kNil) {
        const uint4 *p = reinterpret_cast<const uint4 *>(slab_ptr(g, s) + (lane_id() & 3u) * 8);
        lo = __ldcg(p);
        hi = __ldcg(p + 1);
    }
}

// The k-th set bit of q handed to 4-lane group `gi` in pass `pass` (eight
// groups per pass): returns the lane index holding that group's item, or
// 32 when the pass has fewer items than groups.
__device__ __forceinline__ uint32_t group_item(uint32_t q, uint32_t pass, uint32_t gi)
{
    const uint32_t k = pass * 8 + gi;
    if (k >= (uint32_t)__popc(q))
        return 32;
    return nth_set_bit(q, k);
}

} // namespace mk
