// ConcurrentSet layout (paper, Sec. "Motivation": SlabHash's ConcurrentSet
// beside the ConcurrentMap that the weighted store uses; the paper stores the
// unweighted graphs of BFS and WCC this way).  An unweighted graph whose
// slabs hold 31 destination keys (lanes 0..30) and the next-slab index
// (lane 31): about twice the keys of a map slab's 15 pairs, so the slab
// array, and every traversal that streams it, is about half as large.
//
// The store keeps the map store's conventions: one head slab per bucket of a
// vertex in one allocation located by an exclusive scan of the bucket
// counts, overflow slabs claimed from a bitmap pool, EMPTY and TOMBSTONE
// keys, deleted keys never reused (so free keys exist only in a chain's last
// slab), set semantics with the first occurrence of a repeated pair applied
// (a larger batch is grouped by slab list, as the map store's are: group.cu).
// Inserts, deletes and queries walk eight chains per warp in 4-lane groups,
// each lane reading 32 bytes of a slab (the whole group one 128-byte slab).
// BFS (hop counts, with the smallest-id tight parent) and WCC (smallest-id
// labels) run statically: BFS level by level over a frontier of lists, WCC
// as the map store's static pass (wcc.cu).
#include "mk_host.h"
#include "walk.cuh"
#include "uf.cuh"

#include <algorithm>
#include <cstring>

using namespace mk;

// Kernels of other translation units, launched here unchanged.
constexpr uint32_t kDegBlock = 512;
__global__ void __launch_bounds__(kDegBlock) k_degree(const uint32_t *__restrict__ src, uint64_t n, uint32_t V,
                                                      uint32_t *deg, int *bad);
uint32_t degree_grid(uint64_t n);
__global__ void k_rule(uint32_t *deg, uint32_t V, float per_bucket);
__global__ void k_init_bitmap(uint32_t *bitmap, uint32_t words, uint32_t P);
__global__ void k_fill_buckets(uint32_t *b, uint32_t V, uint32_t nb, const uint32_t *user, int *bad);
__global__ void __launch_bounds__(256) k_check_edges(const uint32_t *__restrict__ src, const uint32_t *__restrict__ dst,
                                                     const uint32_t *__restrict__ w, uint64_t n, uint32_t V,
                                                     DevState *st);

namespace {

constexpr uint32_t kSetKeys = 31; // key lanes 0..30, lane 31 = next

} // namespace

struct mk_set_graph {
    int device = 0;            // the device that was current at its creation
    GView v{};                 // V, H, P, pool_words, vinfo, slabs, bitmap, owner, st (the rest unused)
    uint64_t bytes = 0;
    GroupScratch group;        // staging of inserts and deletes
    // most edges of one grouping, of a delete and of an insert that is not
    // grouped (mk_set_debug_set)
    uint64_t dbg_part = kGroupEdges, dbg_hash[2] = {kHashSetDelete, kHashSetInsert};
    uint32_t *h_pinned = nullptr;
};

// -------------------------------------------------------------- kernels

__global__ void k_set_init_slabs(uint32_t *slabs, uint64_t count)
{
    const uint64_t words = count * 32;
    for (uint64_t i = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; i < words;
         i += (uint64_t)gridDim.x * blockDim.x)
        slabs[i] = (i & 31) == kNextLane ? kNil : kEmptyKey;
}

// vinfo[v] = {first list, bucket count}; owner[list] = v; owner of every
// pool slab = kNil.
__global__ void k_set_init_lists(const uint64_t *off, const uint32_t *buckets, uint32_t V, uint2 *vinfo,
                                 uint32_t *owner, uint64_t H, uint64_t total)
{
    const uint64_t stride = (uint64_t)gridDim.x * blockDim.x;
    const uint32_t lane = lane_id();
    for (uint64_t vb = (blockIdx.x * (uint64_t)blockDim.x + threadIdx.x) & ~31ull; vb < V; vb += stride) {
        const uint32_t v = (uint32_t)vb + lane;
        const uint32_t first = v < V ? (uint32_t)off[v] : 0, nb = v < V ? buckets[v] : 0;
        if (v < V)
            vinfo[v] = make_uint2(first, nb);
        if (nb <= 8)
            for (uint32_t b = 0; b < nb; ++b)
                owner[first + b] = v;
        // a hub's lists are written by its whole warp
        for (uint32_t big = __ballot_sync(kFull, nb > 8); big; big &= big - 1) {
            const uint32_t l = __ffs(big) - 1;
            const uint32_t f = __shfl_sync(kFull, first, l), m = __shfl_sync(kFull, nb, l);
            const uint32_t own = __shfl_sync(kFull, v, l);
            for (uint32_t b = lane; b < m; b += 32)
                owner[f + b] = own;
        }
    }
    for (uint64_t s = H + blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; s < total; s += stride)
        owner[s] = kNil;
}

namespace {

// The list that holds (s, d).
__device__ __forceinline__ uint32_t set_list(const GView &g, uint32_t s, uint32_t d)
{
    const uint2 vi = __ldg(&g.vinfo[s]);
    return vi.x + bucket_of(d, vi.y);
}

// Lanes of the calling lane's 4-lane group in a warp-wide ballot.
__device__ __forceinline__ uint32_t set_group_bits(uint32_t ballot) { return (ballot >> (lane_id() & ~3u)) & 0xFu; }

// Lane s4 of a 4-lane group holds words 8*s4 .. 8*s4+7 of a slab as two
// 16-byte vectors; word 31 (the last of lane 3) is the next index.
__device__ __forceinline__ void set_group_load(const GView &g, uint32_t slab, uint4 &lo, uint4 &hi)
{
    const uint4 *p = reinterpret_cast<const uint4 *>(slab_ptr(g, slab) + (lane_id() & 3u) * 8);
    lo = __ldcg(p);
    hi = __ldcg(p + 1);
}

// Index (0..7) of the lane's first key word equal to k, 8 if none.
__device__ __forceinline__ uint32_t set_first_with(const uint4 &lo, const uint4 &hi, uint32_t k)
{
    const bool last = (lane_id() & 3u) == 3u;
    return lo.x == k   ? 0u
           : lo.y == k ? 1u
           : lo.z == k ? 2u
           : lo.w == k ? 3u
           : hi.x == k ? 4u
           : hi.y == k ? 5u
           : hi.z == k ? 6u
           : (!last && hi.w == k) ? 7u
                                  : 8u;
}

// Inserts d into the list of s with one 4-lane group (go == false: the
// group has nothing to do; every group of the warp calls it in lockstep).
// Walks the whole chain (a present key ends the walk), claims the lowest
// free key of the tail with a CAS (a lost CAS re-reads the slab), or links a
// pool slab holding d with a CAS on the tail's next word (the loser frees
// its slab and follows the winner's).  Returns 1 if d was stored, 0 if it
// was present, or a negative device error code, on the group's lanes.
__device__ __forceinline__ int group_set_insert(const GView &g, bool go, uint32_t s, uint32_t d, uint32_t max_hops,
                                                unsigned long long &loads, unsigned long long &linked)
{
    const uint32_t s4 = lane_id() & 3u, gbase = lane_id() & ~3u;
    bool active = go;
    int res = 0;
    uint32_t slab = go ? set_list(g, s, d) : kNil;
    uint4 lo = make_uint4(kFull, kFull, kFull, kFull), hi = lo;
    if (active)
        set_group_load(g, slab, lo, hi);
    const uint32_t guard_max = 4 * max_hops + 64;
    for (uint32_t guard = 0; __any_sync(kFull, active); ++guard) {
        loads += __popc(__ballot_sync(kFull, active && s4 == 0));
        const uint32_t hits = set_group_bits(__ballot_sync(kFull, active && set_first_with(lo, hi, d) < 8u));
        const uint32_t fk = set_first_with(lo, hi, kEmptyKey);
        const uint32_t frees = set_group_bits(__ballot_sync(kFull, active && fk < 8u));
        const uint32_t nxt = __shfl_sync(kFull, hi.w, gbase + 3);
        // the lowest free key of the group's slab
        bool ok = false;
        if (active && !hits && frees && s4 == (uint32_t)(__ffs(frees) - 1))
            ok = atomicCAS(slab_ptr(g, slab) + 8 * s4 + fk, kEmptyKey, d) == kEmptyKey;
        const bool claimed = set_group_bits(__ballot_sync(kFull, ok)) != 0;
        // a full tail with nothing after it: a pool slab holding d
        const bool grow = active && !hits && !frees && nxt == kNil;
        uint32_t ns = kNil;
        if (grow && s4 == 0)
            ns = alloc_slab_one(g, s * 0x9E3779B9u ^ d ^ (guard << 26));
        ns = __shfl_sync(kFull, ns, gbase);
        uint32_t old = kNil;
        if (grow && ns != kNil) {
            const uint4 e = make_uint4(kEmptyKey, kEmptyKey, kEmptyKey, kEmptyKey);
            const uint4 wlo = s4 == 0 ? make_uint4(d, kEmptyKey, kEmptyKey, kEmptyKey) : e;
            const uint4 whi = s4 == 3u ? make_uint4(kEmptyKey, kEmptyKey, kEmptyKey, kNil) : e;
            uint4 *q = reinterpret_cast<uint4 *>(slab_ptr(g, ns) + s4 * 8);
            __stcg(q, wlo);
            __stcg(q + 1, whi);
            if (s4 == 0)
                g.owner[ns] = s;
            __threadfence();
            if (s4 == 0)
                old = atomicCAS(slab_ptr(g, slab) + kNextLane, kNil, ns);
        }
        old = __shfl_sync(kFull, old, gbase);
        const bool won = grow && ns != kNil && old == kNil;
        linked += __popc(__ballot_sync(kFull, won && s4 == 0));
        if (active) {
            if (hits) {
                active = false; // present already
            } else if (frees) {
                if (claimed) {
                    res = 1;
                    active = false;
                } // else another group took the key: read the slab again
            } else if (nxt != kNil) {
                slab = nxt;
            } else if (ns == kNil) {
                res = kErrPool;
                active = false;
            } else if (won) {
                res = 1;
                active = false;
            } else { // lost the link: give the slab back, follow the winner's
                if (s4 == 0)
                    g.owner[ns] = kNil;
                __threadfence();
                if (s4 == 0)
                    free_slab(g, ns);
                slab = old;
            }
            if (active && guard >= guard_max) {
                res = kErrTimeout;
                active = false;
            }
        }
        if (active)
            set_group_load(g, slab, lo, hi);
    }
    return res;
}

// Deletes d from the list of s with one 4-lane group (layout and lockstep
// as above): the key becomes TOMBSTONE (never reused); the walk stops at the
// key, at the chain's first free key or at its end.  Returns 1 if d was
// removed.
__device__ __forceinline__ int group_set_delete(const GView &g, bool go, uint32_t s, uint32_t d, uint32_t max_hops,
                                                unsigned long long &loads)
{
    const uint32_t s4 = lane_id() & 3u, gbase = lane_id() & ~3u;
    bool active = go;
    int res = 0;
    uint32_t slab = go ? set_list(g, s, d) : kNil;
    uint4 lo = make_uint4(kFull, kFull, kFull, kFull), hi = lo;
    for (uint32_t hop = 0; __any_sync(kFull, active); ++hop) {
        if (active)
            set_group_load(g, slab, lo, hi);
        loads += __popc(__ballot_sync(kFull, active && s4 == 0));
        const uint32_t hk = set_first_with(lo, hi, d);
        const uint32_t hits = set_group_bits(__ballot_sync(kFull, active && hk < 8u));
        const uint32_t frees = set_group_bits(__ballot_sync(kFull, active && set_first_with(lo, hi, kEmptyKey) < 8u));
        const uint32_t nxt = __shfl_sync(kFull, hi.w, gbase + 3);
        bool ok = false;
        if (active && hits && s4 == (uint32_t)(__ffs(hits) - 1))
            ok = atomicCAS(slab_ptr(g, slab) + 8 * s4 + hk, d, kTombKey) == d;
        const bool removed = set_group_bits(__ballot_sync(kFull, ok)) != 0;
        if (active) {
            if (hits) {
                res = removed ? 1 : 0;
                active = false;
            } else if (frees || nxt == kNil || hop + 1 >= max_hops) {
                active = false;
            } else {
                slab = nxt;
            }
        }
    }
    return res;
}

} // namespace

// The lists with many edges in the batch (grouping.many), or all of a batch
// that is not grouped, 32 edges a warp:
// eight 4-lane groups take the first occurrences among them eight at a time,
// so eight chains are walked at once.
template <bool kInsert>
__global__ void __launch_bounds__(256) k_set_update(GView g, GroupView gv, const uint32_t *__restrict__ src,
                                                    const uint32_t *__restrict__ dst, uint64_t all,
                                                    uint8_t *__restrict__ flags, uint32_t max_hops)
{
    const uint32_t lane = lane_id(), gi = lane >> 2;
    const uint64_t warps = ((uint64_t)gridDim.x * blockDim.x) >> 5;
    const uint32_t n = gv.many ? __ldg(&gv.ctr[kGroupMany]) : (uint32_t)all;
    const uint32_t *order = gv.many ? gv.many + __ldg(&gv.ctr[kGroupActive]) : nullptr;
    const uint32_t *tpos = reinterpret_cast<const uint32_t *>(gv.ent);
    unsigned long long loads = 0, linked = 0;
    for (uint64_t q0 = ((blockIdx.x * (uint64_t)blockDim.x + threadIdx.x) >> 5) * 32; q0 < n; q0 += warps * 32) {
        if (__any_sync(kFull, status_hint(g.st) != 0))
            break;
        bool first = false;
        uint32_t i = 0, s = 0, d = 0;
        if (q0 + lane < n) {
            i = order ? order[q0 + lane] : (uint32_t)q0 + lane;
            const uint32_t at = gv.lst[i]; // kNil: an invalid edge, which no grouped list holds
            first = at != kNil && __ldcg(&tpos[at & ~kSlotBit]) == i;
            s = src[i];
            d = dst[i];
        }
        uint8_t mine = 0;
#pragma unroll 1
        for (uint32_t it = 0; it < 4; ++it) {
            const uint32_t who = it * 8 + gi;
            const bool go = __shfl_sync(kFull, first, who);
            const uint32_t ws = __shfl_sync(kFull, s, who), wd = __shfl_sync(kFull, d, who);
            const int r = kInsert ? group_set_insert(g, go, ws, wd, max_hops, loads, linked)
                                  : group_set_delete(g, go, ws, wd, max_hops, loads);
            if (r < 0 && (lane & 3u) == 0)
                set_status(g.st, r);
            // lane L's edge was taken by group L % 8 in step L / 8
            const int rl = __shfl_sync(kFull, r, (lane & 7u) * 4);
            if (lane / 8 == it)
                mine = rl > 0 ? 1 : 0;
        }
        if (flags && mine)
            flags[i] = 1;
    }
    count_add(g.st, kInsert ? kCtrInsertSlabs : kCtrDeleteSlabs, loads);
    count_add(g.st, kCtrInsertNewSlabs, linked);
}

namespace {

// Bit q: the lane's key q of a slab is k (the last lane's eighth word is the
// next index).
__device__ __forceinline__ uint32_t set_keys_with(const uint4 &lo, const uint4 &hi, uint32_t k)
{
    return (lo.x == k ? 1u : 0u) | (lo.y == k ? 2u : 0u) | (lo.z == k ? 4u : 0u) | (lo.w == k ? 8u : 0u) |
           (hi.x == k ? 16u : 0u) | (hi.y == k ? 32u : 0u) | (hi.z == k ? 64u : 0u) |
           ((lane_id() & 3u) != 3u && hi.w == k ? 128u : 0u);
}

using SetMask = unsigned long long; // over a list's edges
static_assert(kSetGroupMax <= 64, "a bit an edge");

} // namespace

// Applies the grouped inserts, one list a 4-lane group, eight a warp, as the
// weighted store's k_apply_insert does (no weights, no logs): the list's
// repeats found among its edges, its chain walked once, its free keys filled
// and pool slabs linked with plain stores.  R-MAT scale 19 load, 8.4 M edges
// into 0.9 M lists, staging included: 720 us with a batch hash set and a CAS
// an edge, 470 so.
__global__ void __launch_bounds__(256, 4) k_set_apply_insert(GView g, GroupView gv, uint8_t *__restrict__ flags,
                                                             uint32_t max_hops)
{
    __shared__ uint2 rows[kGroupLists][kSetGroupMax + 1];    // each list's edges (an odd stride: the lists of a
    __shared__ uint32_t fresh[kGroupLists][kSetGroupMax + 1]; // warp differ in their banks), and its new keys
    const uint32_t lane = lane_id(), s4 = lane & 3u, gbase = lane & ~3u;
    uint2 *row = rows[threadIdx.x >> 2];
    uint32_t *add = fresh[threadIdx.x >> 2];
    const bool dead = read_status(g.st) != 0;
    ListCursor cur = first_lists(g, gv);
    unsigned long long loads = 0, linked = 0;
    while (__any_sync(kFull, cur.at < cur.n)) {
        const uint3 my = next_list(gv, cur, dead);
        const uint32_t L = my.x, c = my.y;
        if (!__any_sync(kFull, c))
            continue;
        uint4 lo = make_uint4(kEmptyKey, kEmptyKey, kEmptyKey, kEmptyKey), hi = lo;
        if (c)
            set_group_load(g, L, lo, hi);
        SetMask news = group_first<SetMask>(gv, c, my.z, row), have = 0;
        uint32_t slab = L, frees = 0;
        bool active = c != 0;
        int err = 0;
        for (uint32_t hop = 0; __any_sync(kFull, active); ++hop) {
            if (active && hop)
                set_group_load(g, slab, lo, hi);
            loads += __popc(__ballot_sync(kFull, active && s4 == 0));
            const bool empty = __shfl_sync(kFull, lo.x, gbase) == kEmptyKey; // keys fill in order
            if (active && !empty)
                for (uint32_t e = 0; e < c; ++e)
                    have |= (SetMask)(set_keys_with(lo, hi, row[e].x) != 0) << e;
            const uint32_t f = group_or(set_keys_with(lo, hi, kEmptyKey) << (8 * s4));
            const uint32_t nxt = __shfl_sync(kFull, hi.w, gbase + 3);
            if (active) {
                frees = f;
                if (f || nxt == kNil) {
                    active = false; // the tail: free keys exist only in the last slab
                } else if (hop + 1 >= max_hops) {
                    err = kErrTimeout;
                    active = false;
                } else {
                    slab = nxt;
                }
            }
        }
        news = err ? 0ull : news & ~group_or(have);
        const uint32_t k = __popcll(news), room = __popc(frees);
        for (uint32_t e = s4; e < c; e += 4)
            if ((news >> e) & 1u)
                add[__popcll(news & ((1ull << e) - 1))] = row[e].x;
        __syncwarp();
#pragma unroll
        for (uint32_t q = 0; q < 8; ++q) {
            const uint32_t p = 8 * s4 + q, r = __popc(frees & ((1u << p) - 1));
            if (((frees >> p) & 1u) && r < k)
                slab_ptr(g, slab)[p] = add[r];
        }
        uint32_t stored = min(k, room), prev = slab;
        for (uint32_t t = 0; __any_sync(kFull, !err && stored < k); ++t) {
            const bool grow = !err && stored < k;
            uint32_t ns = kNil;
            if (grow && s4 == 0)
                ns = alloc_slab_one(g, L * 0x9E3779B9u ^ (t << 24));
            ns = __shfl_sync(kFull, ns, gbase);
            linked += __popc(__ballot_sync(kFull, grow && ns != kNil && s4 == 0));
            if (grow && ns == kNil)
                err = kErrPool;
            if (grow && ns != kNil) {
                uint32_t w[8];
#pragma unroll
                for (uint32_t q = 0; q < 8; ++q) {
                    const uint32_t r = stored + 8 * s4 + q;
                    w[q] = r < k && 8 * s4 + q < kSetKeys ? add[r] : kEmptyKey;
                }
                if (s4 == 3u)
                    w[7] = kNil;
                uint4 *to = reinterpret_cast<uint4 *>(slab_ptr(g, ns) + s4 * 8);
                __stcg(to, make_uint4(w[0], w[1], w[2], w[3]));
                __stcg(to + 1, make_uint4(w[4], w[5], w[6], w[7]));
                if (s4 == 3u) // lane 3 holds the next words, so it links what it wrote before
                    slab_ptr(g, prev)[kNextLane] = ns;
                if (s4 == 0)
                    g.owner[ns] = __ldg(&g.owner[L]);
                prev = ns;
                stored = min(k, stored + kSetKeys);
            }
        }
        if (err && s4 == 0)
            set_status(g.st, err);
        if (flags)
            for (uint32_t e = s4; e < c; e += 4)
                if (((news >> e) & 1u) && (uint32_t)__popcll(news & ((1ull << e) - 1)) < stored)
                    flags[row[e].y] = 1;
    }
    count_add(g.st, kCtrInsertSlabs, loads);
    count_add(g.st, kCtrInsertNewSlabs, linked);
}

// Applies the grouped deletes in the same way.
__global__ void __launch_bounds__(256, 5) k_set_apply_delete(GView g, GroupView gv, uint8_t *__restrict__ flags,
                                                             uint32_t max_hops)
{
    __shared__ uint2 rows[kGroupLists][kSetGroupMax + 1];
    const uint32_t lane = lane_id(), s4 = lane & 3u, gbase = lane & ~3u;
    uint2 *row = rows[threadIdx.x >> 2];
    const bool dead = read_status(g.st) != 0;
    ListCursor cur = first_lists(g, gv);
    unsigned long long loads = 0;
    while (__any_sync(kFull, cur.at < cur.n)) {
        const uint3 my = next_list(gv, cur, dead);
        const uint32_t L = my.x, c = my.y;
        if (!__any_sync(kFull, c))
            continue;
        uint4 lo = make_uint4(kEmptyKey, kEmptyKey, kEmptyKey, kEmptyKey), hi = lo;
        if (c)
            set_group_load(g, L, lo, hi);
        SetMask todo = group_first<SetMask>(gv, c, my.z, row), gone = 0;
        uint32_t slab = L;
        bool active = c != 0;
        for (uint32_t hop = 0; __any_sync(kFull, active); ++hop) {
            if (active && hop)
                set_group_load(g, slab, lo, hi);
            loads += __popc(__ballot_sync(kFull, active && s4 == 0));
            SetMask hit = 0;
            if (active)
                for (SetMask left = todo; left; left &= left - 1) {
                    const uint32_t e = __ffsll((long long)left) - 1, at = set_keys_with(lo, hi, row[e].x);
                    if (at) {
                        hit |= 1ull << e;
                        slab_ptr(g, slab)[8 * s4 + __ffs(at) - 1] = kTombKey;
                    }
                }
            hit = group_or(hit);
            const uint32_t f = group_or(set_keys_with(lo, hi, kEmptyKey));
            const uint32_t nxt = __shfl_sync(kFull, hi.w, gbase + 3);
            todo &= ~hit;
            gone |= hit;
            if (active) {
                if (!todo || f || nxt == kNil || hop + 1 >= max_hops)
                    active = false;
                else
                    slab = nxt;
            }
        }
        if (flags)
            for (uint32_t e = s4; e < c; e += 4)
                if ((gone >> e) & 1u)
                    flags[row[e].y] = 1;
    }
    count_add(g.st, kCtrDeleteSlabs, loads);
}

// Queries: bit i % 32 of word i / 32 is set when edge i is present.  One
// warp answers 32 consecutive queries: every lane first finds its own
// query's list (32 gathers in flight), then the warp walks eight chains at
// a time, one per 4-lane group, each lane loading 8 consecutive words of
// the slab as two 16-byte vectors (the group's last lane holds the next
// index in its last word).
__global__ void __launch_bounds__(256) k_set_query(GView g, const uint32_t *__restrict__ src,
                                                   const uint32_t *__restrict__ dst, uint64_t n,
                                                   uint32_t *__restrict__ bitmap, uint32_t max_hops)
{
    constexpr uint32_t G = 4, W = 8, kGroups = 8;
    const uint32_t lane = lane_id(), gi = lane / G, sub = lane % G;
    const uint32_t gmask = 0xFu << (gi * G);
    const uint64_t warps = ((uint64_t)gridDim.x * blockDim.x) >> 5;
    unsigned long long loads = 0;
    for (uint64_t q0 = ((blockIdx.x * (uint64_t)blockDim.x + threadIdx.x) >> 5) * 32; q0 < n; q0 += warps * 32) {
        const uint64_t q = q0 + lane;
        uint32_t my_d = kNil, my_head = kNil;
        bool bad = false;
        if (q < n) {
            const uint32_t s = __ldg(src + q);
            my_d = __ldg(dst + q);
            if (s < g.V && my_d < g.V)
                my_head = set_list(g, s, my_d);
            else
                bad = true;
        }
        if (__ballot_sync(kFull, bad) && lane == 0)
            set_status(g.st, kErrInvalid);
        uint32_t word_bits = 0;
#pragma unroll 1
        for (uint32_t it = 0; it < 32 / kGroups; ++it) {
            const uint32_t who = it * kGroups + gi;
            const uint32_t d = __shfl_sync(kFull, my_d, who);
            uint32_t slab = __shfl_sync(kFull, my_head, who);
            bool active = slab != kNil, found = false;
            for (uint32_t hop = 0; __any_sync(kFull, active); ++hop) {
                loads += __popc(__ballot_sync(kFull, active && sub == 0));
                uint4 a = make_uint4(kFull, kFull, kFull, kFull), b = a;
                if (active) {
                    const uint4 *v = reinterpret_cast<const uint4 *>(slab_ptr(g, slab) + sub * W);
                    a = __ldg(v);
                    b = __ldg(v + 1);
                }
                const uint32_t w[W] = {a.x, a.y, a.z, a.w, b.x, b.y, b.z, b.w};
                bool hit = false, emp = false;
#pragma unroll
                for (uint32_t k = 0; k < W; ++k)
                    if (sub * W + k < kSetKeys) {
                        hit |= active && w[k] == d;
                        emp |= active && w[k] == kEmptyKey;
                    }
                const uint32_t hm = __ballot_sync(kFull, hit) & gmask;
                const uint32_t em = __ballot_sync(kFull, emp) & gmask;
                const uint32_t nxt = __shfl_sync(kFull, b.w, gi * G + G - 1);
                if (hm)
                    found = true;
                if (active && (hm || em || nxt == kNil || hop >= max_hops))
                    active = false;
                else if (active)
                    slab = nxt;
            }
            const uint32_t fb = __ballot_sync(kFull, sub == 0 && found);
#pragma unroll
            for (uint32_t k = 0; k < kGroups; ++k)
                if (fb & (1u << (k * G)))
                    word_bits |= 1u << (it * kGroups + k);
        }
        if (lane == 0 && q0 < n)
            bitmap[q0 / 32] = word_bits;
    }
    count_add(g.st, kCtrQuerySlabs, loads);
}

// One BFS level over a frontier of <list, source>, one list per 4-lane group
// (eight lists per warp in flight, so a hub's buckets spread over many
// groups, and the next eight being read); each lane tests the eight keys of
// its 32 bytes of a slab at once.  A destination still unreached gets level +
// 1 with a CAS and its lists join the next frontier through the warp's
// staging buffer.  The parents come out of the same pass: an edge read into a
// vertex of the next level is tight, so an atomicMin of the list's source
// leaves the smallest one.  The frontier sizes live on the device in three
// rotating counters (this level reads cnt[L % 3], appends to cnt[(L + 1) % 3]
// and clears cnt[(L + 2) % 3], the input of the level before), so several
// levels go out without the host.  What bounds a large level is the chain of
// a list (distances, CAS, bucket ranges), at 100 G gathers/s: R-MAT scale 19,
// 8 M edges, 156 us a search, 165 with an append to the frontier a slab step
// (a read of the parent before its atomicMin made it 174).
__global__ void __launch_bounds__(256, 4) k_set_bfs_level(GView g, const uint2 *__restrict__ front, uint2 *next,
                                                       uint32_t *cnt, uint32_t *dist, uint32_t *parent,
                                                       uint32_t level, uint32_t max_hops)
{
    __shared__ FrontierSmem<8> bq;
    const uint32_t lane = lane_id(), s4 = lane & 3u, gbase = lane & ~3u;
    const uint32_t n = __ldcg(&cnt[level % 3]);
    uint32_t *next_count = &cnt[(level + 1) % 3];
    int *overflow = (int *)&cnt[3]; // a vertex is queued once, so its lists fit
    if (blockIdx.x == 0 && threadIdx.x == 0)
        cnt[(level + 2) % 3] = 0;
    if ((blockIdx.x * (uint64_t)blockDim.x) >> 2 >= n)
        return;
    frontier_init(bq);
    const uint64_t groups = ((uint64_t)gridDim.x * blockDim.x) >> 2;
    const uint64_t g0 = (blockIdx.x * (uint64_t)blockDim.x + threadIdx.x) >> 2;
    unsigned long long loads = 0;
    auto entry = [&](uint64_t k) { return k < n ? __ldcg(&front[k]) : make_uint2(kNil, 0u); };
    auto load = [&](uint32_t slab, uint4 &lo, uint4 &hi) {
        lo = hi = make_uint4(kFull, kFull, kFull, kFull);
        if (slab != kNil)
            set_group_load(g, slab, lo, hi);
    };
    // the group's next list is read while the current one is worked on
    uint2 e = entry(g0), ne = entry(g0 + groups);
    uint4 lo, hi;
    load(e.x, lo, hi);
    // the warp's eight groups move together: `wb` is its first group's index
    for (uint64_t wb = g0 & ~7ull; wb < n; wb += groups) {
        const uint2 nne = entry(wb + (g0 & 7u) + 2 * groups);
        uint4 nlo, nhi;
        load(ne.x, nlo, nhi);
        uint32_t slab = e.x;
        const uint32_t u = e.y; // the list's source, at this level
        bool active = slab != kNil;
        for (uint32_t hop = 0; __any_sync(kFull, active); ++hop) {
            if (hop)
                load(active ? slab : kNil, lo, hi);
            loads += __popc(__ballot_sync(kFull, active && s4 == 0));
            const uint32_t wv[8] = {lo.x, lo.y, lo.z, lo.w, hi.x, hi.y, hi.z, hi.w};
            uint32_t cur[8];
            bool key[8];
#pragma unroll
            for (int q = 0; q < 8; ++q) {
                key[q] = active && s4 * 8 + q < kSetKeys && wv[q] < kTombKey;
                cur[q] = key[q] ? __ldcg(&dist[wv[q]]) : 0u;
            }
            bool grab[8], any = false;
#pragma unroll
            for (int q = 0; q < 8; ++q) {
                grab[q] = key[q] && cur[q] == kNil && atomicCAS(&dist[wv[q]], kNil, level + 1) == kNil;
                any = any || grab[q];
            }
            // every edge into a vertex of the next level is tight: the
            // smallest such source is the parent (dist only moves from
            // unreached to level + 1 during this launch, so a destination
            // read as unreached is at level + 1 now, whoever took it)
#pragma unroll
            for (int q = 0; q < 8; ++q)
                if (key[q] && (cur[q] == kNil || cur[q] == level + 1))
                    atomicMin(&parent[wv[q]], u);
            const uint32_t nxt = __shfl_sync(kFull, hi.w, gbase + 3);
            if (__any_sync(kFull, any)) {
                uint2 vi[8];
#pragma unroll
                for (int q = 0; q < 8; ++q)
                    vi[q] = grab[q] ? __ldg(&g.vinfo[wv[q]]) : make_uint2(0, 0);
                enqueue_lists<8>(bq, wv, grab, vi, next, next_count, g.H, overflow);
            }
            if (active) {
                if (nxt == kNil || hop + 1 >= max_hops)
                    active = false;
                else
                    slab = nxt;
            }
        }
        e = ne;
        ne = nne;
        lo = nlo;
        hi = nhi;
    }
    frontier_flush(bq, next, next_count, g.H, overflow);
    count_add(g.st, kCtrRelaxSlabs, loads);
}

// dist / parent start values; the first frontier is the source's lists.
__global__ void k_set_bfs_init(GView g, uint32_t *dist, uint32_t *parent, uint32_t source, uint2 *front,
                               uint32_t *cnt)
{
    const uint32_t v = blockIdx.x * blockDim.x + threadIdx.x;
    const uint2 vi = __ldg(&g.vinfo[source]);
    if (v < g.V) {
        dist[v] = v == source ? 0u : kNil;
        parent[v] = v == source ? source : kNil;
    }
    for (uint32_t i = v; i < vi.y; i += gridDim.x * blockDim.x)
        front[i] = make_uint2(vi.x + i, source);
    if (v == 0) {
        cnt[0] = vi.y;
        cnt[1] = cnt[2] = cnt[3] = 0;
    }
}

__global__ void k_set_pool_used(const DevState *st, unsigned long long *out)
{
    long long t = 0;
    for (uint32_t i = 0; i < kSlots; ++i)
        t += st->pool_used[i];
    *out = (unsigned long long)t;
}

// ------------------------------------------------------------- host side

namespace {

mk_status set_alloc(mk_set_graph *g, void **p, size_t bytes, cudaStream_t s)
{
    *p = nullptr;
    if (!bytes)
        return MK_OK;
    const cudaError_t e = pool_alloc_kept(p, bytes, s);
    if (e != cudaSuccess)
        return e == cudaErrorMemoryAllocation ? MK_ERR_NO_MEMORY : MK_ERR_CUDA;
    g->bytes += bytes;
    return MK_OK;
}

uint32_t set_grid(uint64_t items_per_warp32)
{
    return std::min<uint32_t>(grid_for(std::max<uint64_t>(items_per_warp32, 1) * 32, 256), num_sms() * 32);
}

// Inserts or deletes n edges, in parts of at most dbg_part (a batch of more
// is checked whole first, so that it is still rejected whole).
template <bool kInsert>
mk_status set_apply(mk_set_graph *g, const uint32_t *d_src, const uint32_t *d_dst, uint64_t n, uint8_t *d_flags,
                    cudaStream_t s)
{
    if (d_flags)
        MK_CUDA(cudaMemsetAsync(d_flags, 0, n, s));
    if (n > g->dbg_part)
        k_check_edges<<<grid_for(n, 256), 256, 0, s>>>(d_src, d_dst, nullptr, n, g->v.V, g->v.st);
    for (uint64_t at = 0; at < n; at += g->dbg_part) {
        const uint64_t m = std::min(g->dbg_part, n - at);
        const uint32_t *src = d_src + at, *dst = d_dst + at;
        uint8_t *fl = d_flags ? d_flags + at : nullptr;
        GroupView gv{};
        int launches = 0;
        const bool hash = m <= g->dbg_hash[kInsert];
        MK_CUDA(group_reserve(g->group, m, g->v.H, s, &g->bytes));
        MK_CUDA(hash ? hash_batch(g->v, g->group, src, dst, nullptr, m, nullptr, s, &gv, &launches)
                     : group_batch(g->v, g->group, src, dst, nullptr, m, kSetGroupMax, s, &gv, &launches));
        k_set_update<kInsert><<<set_grid((m + 31) / 32), 256, 0, s>>>(g->v, gv, src, dst, m, fl, g->v.P + 2);
        if (hash) {
            MK_CUDA(cudaGetLastError());
            continue;
        }
        const uint64_t lists = group_dense(g->v.H, m) ? g->v.H : m;
        const uint32_t grid = (uint32_t)std::min<uint64_t>((lists + kGroupLists - 1) / kGroupLists,
                                                           (uint64_t)num_sms() * (kInsert ? 4 : 5));
        if (kInsert)
            k_set_apply_insert<<<grid, 256, 0, s>>>(g->v, gv, fl, g->v.P + 2);
        else
            k_set_apply_delete<<<grid, 256, 0, s>>>(g->v, gv, fl, g->v.P + 2);
        MK_CUDA(cudaGetLastError());
    }
    return MK_OK;
}


} // namespace

extern "C" {

mk_status mk_set_bucket_rule(uint32_t V, const uint32_t *d_src, uint64_t n, float load_factor, uint32_t *d_buckets,
                             void *stream)
{
    if (V == 0 || !d_buckets || (n > 0 && !d_src) || !(load_factor > 0.f) || load_factor > 1.f)
        return MK_ERR_INVALID_ARG;
    cudaStream_t s = (cudaStream_t)stream;
    int *d_bad = nullptr;
    MK_CUDA(pool_alloc((void **)&d_bad, sizeof(int), s));
    MK_CUDA(cudaMemsetAsync(d_bad, 0, sizeof(int), s));
    MK_CUDA(cudaMemsetAsync(d_buckets, 0, (size_t)V * 4, s));
    if (n)
        k_degree<<<degree_grid(n), kDegBlock, 0, s>>>(d_src, n, V, d_buckets, d_bad);
    k_rule<<<grid_for(V, 256), 256, 0, s>>>(d_buckets, V, load_factor * (float)kSetKeys);
    int bad = 0;
    MK_CUDA(cudaMemcpyAsync(&bad, d_bad, sizeof(int), cudaMemcpyDeviceToHost, s));
    MK_CUDA(cudaFreeAsync(d_bad, s));
    MK_CUDA(cudaStreamSynchronize(s));
    return bad ? MK_ERR_INVALID_ARG : MK_OK;
}

mk_status mk_set_destroy(mk_set_graph *g)
{
    if (!g)
        return MK_ERR_INVALID_ARG;
    const DeviceScope on(g->device); // as mk_graph_destroy
    cudaDeviceSynchronize();
    pool_free((void *)g->v.vinfo, nullptr);
    pool_free((void *)g->v.slabs, nullptr);
    pool_free((void *)g->v.bitmap, nullptr);
    pool_free((void *)g->v.owner, nullptr);
    pool_free((void *)g->v.st, nullptr);
    group_release(g->group, &g->bytes, nullptr);
    if (g->h_pinned)
        cudaFreeHost(g->h_pinned);
    pool_settle(g->bytes); // of the arrays freed above
    delete g;
    return MK_OK;
}

mk_status mk_set_create(uint32_t V, uint64_t edge_capacity_hint, uint32_t buckets, const uint32_t *d_bucket_per_vertex,
                        void *stream, mk_set_graph **out)
{
    if (!out || V == 0 || V > 0xFFFFFFFDu)
        return MK_ERR_INVALID_ARG;
    *out = nullptr;
    cudaStream_t s = (cudaStream_t)stream;
    int device = 0;
    MK_CUDA(cudaGetDevice(&device));
    mk_set_graph *g = new mk_set_graph;
    g->device = device;
    g->v.V = V;
    uint32_t *d_b = nullptr;
    uint64_t *d_off = nullptr;
    void *d_tmp = nullptr;
    int *d_bad = nullptr;
    mk_status st = MK_OK;
    auto fail = [&](mk_status code) {
        pool_free(d_b, s);
        pool_free(d_off, s);
        pool_free(d_tmp, s);
        pool_free(d_bad, s);
        mk_set_destroy(g);
        return code;
    };
    if (pool_alloc((void **)&d_b, (size_t)V * 4, s) != cudaSuccess ||
        pool_alloc((void **)&d_off, ((size_t)V + 1) * 8, s) != cudaSuccess ||
        pool_alloc((void **)&d_bad, sizeof(int), s) != cudaSuccess ||
        pool_alloc(&d_tmp, exclusive_scan_scratch_bytes(V + 1), s) != cudaSuccess)
        return fail(MK_ERR_NO_MEMORY);
    cudaMemsetAsync(d_bad, 0, sizeof(int), s);
    k_fill_buckets<<<grid_for(V, 256), 256, 0, s>>>(d_b, V, buckets ? buckets : 1, d_bucket_per_vertex, d_bad);
    if (exclusive_scan_u32_u64(d_b, d_off, V, d_tmp, s, nullptr) != cudaSuccess)
        return fail(MK_ERR_CUDA);
    // H = last offset + last bucket count
    uint64_t last_off = 0;
    uint32_t last_b = 0;
    int bad = 0;
    if (cudaMemcpyAsync(&last_off, d_off + V - 1, 8, cudaMemcpyDeviceToHost, s) != cudaSuccess ||
        cudaMemcpyAsync(&last_b, d_b + V - 1, 4, cudaMemcpyDeviceToHost, s) != cudaSuccess ||
        cudaMemcpyAsync(&bad, d_bad, sizeof(int), cudaMemcpyDeviceToHost, s) != cudaSuccess ||
        cudaStreamSynchronize(s) != cudaSuccess)
        return fail(MK_ERR_CUDA);
    if (bad)
        return fail(MK_ERR_INVALID_ARG);
    const uint64_t H = last_off + last_b;
    uint64_t P = edge_capacity_hint / kSetKeys + H / 8 + 1024;
    P = (P + 31) / 32 * 32;
    if (H + P >= 0xFFFFFFF0ull)
        return fail(MK_ERR_INVALID_ARG);
    g->v.H = (uint32_t)H;
    g->v.P = (uint32_t)P;
    g->v.pool_words = (uint32_t)(P / 32);
    if ((st = set_alloc(g, (void **)&g->v.vinfo, (size_t)V * 8, s)) != MK_OK ||
        (st = set_alloc(g, (void **)&g->v.slabs, (H + P) * 128, s)) != MK_OK ||
        (st = set_alloc(g, (void **)&g->v.bitmap, (size_t)g->v.pool_words * 4, s)) != MK_OK ||
        (st = set_alloc(g, (void **)&g->v.owner, (H + P) * 4, s)) != MK_OK ||
        (st = set_alloc(g, (void **)&g->v.st, sizeof(DevState), s)) != MK_OK)
        return fail(st);
    uint2 *vinfo = (uint2 *)g->v.vinfo;
    if (cudaMallocHost((void **)&g->h_pinned, 64) != cudaSuccess)
        return fail(MK_ERR_NO_MEMORY);
    cudaMemsetAsync(g->v.st, 0, sizeof(DevState), s);
    k_set_init_slabs<<<std::min<uint64_t>(grid_for((H + P) * 32, 256), 65535), 256, 0, s>>>(g->v.slabs, H + P);
    k_set_init_lists<<<std::min<uint64_t>(grid_for(std::max<uint64_t>(V, P), 256), 65535), 256, 0, s>>>(
        d_off, d_b, V, vinfo, g->v.owner, H, H + P);
    k_init_bitmap<<<grid_for(g->v.pool_words, 256), 256, 0, s>>>(g->v.bitmap, g->v.pool_words, (uint32_t)P);
    if (cudaGetLastError() != cudaSuccess || cudaStreamSynchronize(s) != cudaSuccess)
        return fail(MK_ERR_CUDA);
    pool_free(d_b, s);
    pool_free(d_off, s);
    pool_free(d_tmp, s);
    pool_free(d_bad, s);
    *out = g;
    return MK_OK;
}

mk_status mk_set_insert_batch(mk_set_graph *g, const uint32_t *d_src, const uint32_t *d_dst, uint64_t n,
                              uint8_t *d_inserted, void *stream)
{
    if (!g || (n && (!d_src || !d_dst)) || n >= 0xFFFFFFFFull)
        return MK_ERR_INVALID_ARG;
    if (!n)
        return MK_OK;
    return set_apply<true>(g, d_src, d_dst, n, d_inserted, (cudaStream_t)stream);
}

mk_status mk_set_delete_batch(mk_set_graph *g, const uint32_t *d_src, const uint32_t *d_dst, uint64_t n,
                              uint8_t *d_deleted, void *stream)
{
    if (!g || (n && (!d_src || !d_dst)) || n >= 0xFFFFFFFFull)
        return MK_ERR_INVALID_ARG;
    if (!n)
        return MK_OK;
    return set_apply<false>(g, d_src, d_dst, n, d_deleted, (cudaStream_t)stream);
}

mk_status mk_set_query_batch(mk_set_graph *g, const uint32_t *d_src, const uint32_t *d_dst, uint64_t n,
                             uint32_t *d_bitmap, void *stream)
{
    if (!g || (n && (!d_src || !d_dst || !d_bitmap)))
        return MK_ERR_INVALID_ARG;
    if (!n)
        return MK_OK;
    cudaStream_t s = (cudaStream_t)stream;
    k_set_query<<<set_grid((n + 31) / 32), 256, 0, s>>>(g->v, d_src, d_dst, n, d_bitmap, g->v.P + 2);
    MK_CUDA(cudaGetLastError());
    return MK_OK;
}

mk_status mk_set_bfs(mk_set_graph *g, uint32_t source, uint32_t *d_dist, uint32_t *d_parent, void *stream)
{
    if (!g || source >= g->v.V || !d_dist || !d_parent)
        return MK_ERR_INVALID_ARG;
    cudaStream_t s = (cudaStream_t)stream;
    const uint32_t V = g->v.V;
    const uint64_t H = g->v.H;
    // levels go out in groups; the host reads the frontier size once a group
    constexpr uint32_t kGroup = 6;
    uint2 *front[2] = {nullptr, nullptr};
    uint32_t *cnt = nullptr;
    MK_CUDA(pool_alloc((void **)&front[0], H * 8, s));
    MK_CUDA(pool_alloc((void **)&front[1], H * 8, s));
    MK_CUDA(pool_alloc((void **)&cnt, 16, s));
    k_set_bfs_init<<<grid_for(V, 256), 256, 0, s>>>(g->v, d_dist, d_parent, source, front[0], cnt);
    const uint32_t grid = (uint32_t)num_sms() * 8;
    mk_status st = MK_OK;
    for (uint32_t level = 0;;) {
        if (level > V + kGroup) {
            st = MK_ERR_TIMEOUT;
            break;
        }
        for (uint32_t i = 0; i < kGroup; ++i, ++level)
            k_set_bfs_level<<<grid, 256, 0, s>>>(g->v, front[level & 1], front[(level + 1) & 1], cnt, d_dist,
                                                 d_parent, level, g->v.P + 2);
        if (cudaMemcpyAsync(g->h_pinned, cnt + level % 3, 4, cudaMemcpyDeviceToHost, s) != cudaSuccess ||
            cudaStreamSynchronize(s) != cudaSuccess) {
            st = MK_ERR_CUDA;
            break;
        }
        if (g->h_pinned[0] == 0)
            break;
    }
    cudaFreeAsync(front[0], s);
    cudaFreeAsync(front[1], s);
    cudaFreeAsync(cnt, s);
    return st;
}

mk_status mk_set_wcc(mk_set_graph *g, uint32_t *d_label, void *stream)
{
    if (!g || !d_label)
        return MK_ERR_INVALID_ARG;
    cudaStream_t s = (cudaStream_t)stream;
    const uint32_t V = g->v.V;
    // the forest (and the labels), the giant tree's bitmap, its root and the
    // failure flag in one block
    const size_t words = (size_t)V + ((size_t)V + 31) / 32 + 2;
    uint32_t *p = nullptr;
    MK_CUDA(pool_alloc((void **)&p, words * 4, s));
    uint32_t *bits = p + V, *ctr = p + words - 2;
    int launches = 0;
    cudaError_t e = cudaMemsetAsync(ctr, 0, 8, s);
    if (e == cudaSuccess)
        e = static_components(g->v, true, p, d_label, bits, ctr, (int *)(ctr + 1), s, &launches);
    cudaFreeAsync(p, s);
    return e == cudaSuccess ? MK_OK : MK_ERR_CUDA;
}

mk_status mk_set_stats(mk_set_graph *g, uint64_t *h_lists, uint64_t *h_slabs_in_use, uint64_t *h_device_bytes,
                       void *stream)
{
    if (!g)
        return MK_ERR_INVALID_ARG;
    cudaStream_t s = (cudaStream_t)stream;
    unsigned long long *d = nullptr;
    MK_CUDA(pool_alloc((void **)&d, 8, s));
    k_set_pool_used<<<1, 1, 0, s>>>(g->v.st, d);
    unsigned long long used = 0;
    const cudaError_t e1 = cudaMemcpyAsync(&used, d, 8, cudaMemcpyDeviceToHost, s);
    cudaFreeAsync(d, s);
    if (e1 != cudaSuccess || cudaStreamSynchronize(s) != cudaSuccess)
        return MK_ERR_CUDA;
    if (h_lists)
        *h_lists = g->v.H;
    if (h_slabs_in_use)
        *h_slabs_in_use = g->v.H + used;
    if (h_device_bytes)
        *h_device_bytes = g->bytes;
    return MK_OK;
}

mk_status mk_set_debug_set(mk_set_graph *g, int knob, uint64_t value)
{
    if (!g || (knob != MK_DEBUG_PART_EDGES && knob != MK_DEBUG_HASH_EDGES))
        return MK_ERR_INVALID_ARG;
    if (knob == MK_DEBUG_PART_EDGES) {
        g->dbg_part = part_edges(value);
    } else {
        g->dbg_hash[0] = hash_edges(value, kHashSetDelete);
        g->dbg_hash[1] = hash_edges(value, kHashSetInsert);
    }
    return MK_OK;
}

mk_status mk_set_last_error(mk_set_graph *g)
{
    if (!g)
        return MK_ERR_INVALID_ARG;
    if (cudaDeviceSynchronize() != cudaSuccess)
        return MK_ERR_CUDA;
    int st = 0;
    MK_CUDA(cudaMemcpy(&st, &g->v.st->status, sizeof(int), cudaMemcpyDeviceToHost));
    if (st != 0)
        MK_CUDA(cudaMemset(&g->v.st->status, 0, sizeof(int)));
    return st;
}

} // extern "C"
