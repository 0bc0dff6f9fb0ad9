// Grouping of a batch's edges by slab list (group.cu), shared by the two
// stores' inserts and deletes.
#pragma once

#include "mk_device.cuh"

namespace mk {

// Most edges of one list that a 4-lane group applies by itself: about twice
// the load-factor rule's mean for a list (10 edges of the map layout, 22 of the
// set's).
constexpr uint32_t kGroupMax = 32, kSetGroupMax = 64;
// Marks a hash-set index in GroupView::lst (an edge of a list with more); no
// list has it (2^31 head slabs are 275 GB).
constexpr uint32_t kSlotBit = 0x80000000u;

// What the kernels that apply a grouped batch read.  The edges of list L sit
// at ent[slot[L].y .. + slot[L].x) as <dst, batch position>, in no order, when
// they are at most `most`; otherwise that range holds a hash set of their
// batch positions (2 * slot[L].x words, kNil free) as k_dedup keeps one for a
// whole batch, lst[i] of each of them is its word's index with kSlotBit, and their batch
// positions are the ctr[kGroupMany] words at many[ctr[kGroupActive]].
struct GroupView {
    uint2 *slot;           // per list <edges of this batch, their offset>; the count is 0 between calls
    const uint2 *ent;
    const uint32_t *lst;
    const uint32_t *many;  // null: a batch that is not grouped (hash_batch)
    const uint32_t *alist; // lists with edges, or null when every list is to be looked at
    const uint32_t *ctr;
    uint32_t most;
};
enum { kGroupActive = 0, kGroupCursor = 1, kGroupMany = 2, kGroupWords = 4 };

// Staging arrays of one store, grown on demand: two allocations, at ent (the
// per-edge arrays) and at slot (the lists' counts, then ctr).
struct GroupScratch {
    uint64_t cap = 0;
    uint32_t lists = 0;
    uint32_t *lst = nullptr, *alist = nullptr, *ctr = nullptr;
    uint8_t *rank = nullptr;
    uint2 *ent = nullptr, *slot = nullptr;
};

// Most edges of one grouping (indexes into a hash set, two words an edge,
// have to tell from none).
constexpr uint64_t kGroupEdges = (1ull << 30) - 1;
inline uint64_t part_edges(uint64_t debug) { return debug && debug < kGroupEdges ? debug : kGroupEdges; }

// Whether every list is looked at (and the ranges of the entries follow the
// lists, so that the slabs are streamed in address order), or the lists with
// edges are collected first.
inline bool group_dense(uint32_t H, uint64_t n) { return n >= 4 * (uint64_t)H; }

// Grows the arrays to n edges over H lists (synchronises s when it does);
// *bytes follows what is held.  cudaErrorMemoryAllocation when it cannot.
cudaError_t group_reserve(GroupScratch &gs, uint64_t n, uint32_t H, cudaStream_t s, uint64_t *bytes);
void group_release(GroupScratch &gs, uint64_t *bytes, cudaStream_t s);

// Validates and groups n edges (w nullable, a weight of 0 is invalid), lists of
// up to `most` edges apart from the others, and fills *gv for the kernels launched after it on s.  An invalid edge sets the
// graph's status.  *launches counts the kernels.  The kernel that applies the
// batch must set every active list's count back to 0.
cudaError_t group_batch(const GView &g, GroupScratch &gs, const uint32_t *src, const uint32_t *dst, const uint32_t *w,
                        uint64_t n, uint32_t most, cudaStream_t s, GroupView *gv, int *launches);

// Batches of at most this many edges are not grouped: k_dedup finds their first
// occurrences in a hash set, and the kernels for lists with many edges take all
// of them.  Three launches instead of five, and what is left to do for an edge,
// one search of a chain, gains little from its list's other edges.  us, grouped
// and so, R-MAT scale 17, of 2^20 edges scale 20 and of 2^22 scale 21:
//   deletes of 2^4 / 2^12 / 2^16 / 2^18 / 2^20 / 2^22 edges
//     26 / 36 / 47 / 66 / 148 / 516 and 15 / 25 / 29 / 49 / 123 / 508
//   set deletes 25 / 32 / 39 / 61 / 133 / 414 and 16 / 27 / 31 / 53 / 123 / 465
//   set inserts of 2^4 / 2^12 / 2^16 / 2^18 26 / 37 / 48 / 62 and 19 / 33 / 41 / 69
//   inserts of 1 / 16 / 32 / 2^8 27 / 27 / 28 / 29 and 17 / 21 / 30 / 35: those
//     fill their lists' tails in order, which the other form does one by one
constexpr uint64_t kHashDelete = 1ull << 20, kHashInsert = 16, kHashSetInsert = 1ull << 16, kHashSetDelete = 1ull << 20;
inline uint64_t hash_edges(uint64_t debug, uint64_t most) { return debug ? debug - 1 : most; }

// Words of such a batch's hash set: kHashSpread an edge within 16 MB and what
// the arrays hold, at least two.  (Arrays that are grown for a batch of this
// size get room for kHashRoom times its edges; they are never grown for the
// spread alone, so that a batch that fits neither allocates nor waits.)  A warp
// waits for its longest probe: 2^16 deletes on scale 17 take 53, 39 and 37 us
// with 2, 4 and 16 words.
constexpr uint64_t kHashSpread = 16, kHashWords = 1ull << 22, kHashRoom = 2;
inline uint32_t hash_words(const GroupScratch &gs, uint64_t n)
{
    const uint64_t most = kHashWords < 2 * gs.cap ? kHashWords : 2 * gs.cap;
    const uint64_t words = kHashSpread * n < most ? kHashSpread * n : most;
    return (uint32_t)(words < 2 * n ? 2 * n : words);
}

// Validates n edges of such a batch as group_batch does, and fills *gv with
// their hash set alone: many is null, lst[i] the index of edge i's word among
// those at ent, kNil for an invalid edge; gs holds n edges or more.  log
// (nullable) gets n words of all-ones (update.cu).
cudaError_t hash_batch(const GView &g, GroupScratch &gs, const uint32_t *src, const uint32_t *dst, const uint32_t *w,
                       uint64_t n, unsigned long long *log, cudaStream_t s, GroupView *gv, int *launches);

// Hash of a destination among the 2c words of a list's hash set.
__device__ __forceinline__ uint32_t group_hash(uint32_t d, uint32_t words)
{
    return (uint32_t)(((unsigned long long)hash32(d ^ 0x85ebca6bu) * words) >> 32);
}

// Lists a 256-thread block applies at a time (one a 4-lane group).
constexpr uint32_t kGroupLists = 64;

// The lists of an apply kernel's steps, one a group and step: the list is
// read two steps ahead, its count and range one step ahead.
struct ListCursor {
    uint64_t at, step;
    uint32_t n, L, L1;
    uint2 sl;
};

__device__ __forceinline__ uint32_t list_at(const GroupView &gv, uint64_t k, uint32_t n)
{
    return k < n ? (gv.alist ? __ldg(&gv.alist[k]) : (uint32_t)k) : kNil;
}

__device__ __forceinline__ ListCursor first_lists(const GView &g, const GroupView &gv)
{
    ListCursor c;
    c.n = gv.alist ? __ldg(&gv.ctr[kGroupActive]) : g.H;
    c.at = (blockIdx.x * (uint64_t)blockDim.x + threadIdx.x) >> 2;
    c.step = ((uint64_t)gridDim.x * blockDim.x) >> 2;
    c.L = list_at(gv, c.at, c.n);
    c.L1 = list_at(gv, c.at + c.step, c.n);
    c.sl = c.L != kNil ? gv.slot[c.L] : make_uint2(0, 0);
    return c;
}

// <list, edges, offset> of the calling lane's group, kNil and 0 without work;
// the list's count is set back.  Called by the full warp.
__device__ __forceinline__ uint3 next_list(const GroupView &gv, ListCursor &c, bool dead)
{
    const uint32_t L = c.L;
    const uint2 sl = c.sl;
    c.at += c.step;
    c.L = c.L1;
    c.L1 = list_at(gv, c.at + c.step, c.n);
    c.sl = c.L != kNil ? gv.slot[c.L] : make_uint2(0, 0);
    __syncwarp();
    if (sl.x && (lane_id() & 3u) == 0)
        gv.slot[L].x = 0;
    const bool mine = sl.x != 0 && sl.x <= gv.most && !dead;
    return make_uint3(mine ? L : kNil, mine ? sl.x : 0u, sl.y);
}

// Bits of the four lanes of a group together.
template <typename M>
__device__ __forceinline__ M group_or(M m)
{
    m |= __shfl_xor_sync(kFull, m, 1);
    return m | __shfl_xor_sync(kFull, m, 2);
}

// Entries of the group's list in its shared-memory row, and which of them
// are the first of their destination in batch order, as a mask over entries
// (the same on the group's four lanes; a bit for each of gv.most).  Every lane
// of the warp calls it.
template <typename M>
__device__ __forceinline__ M group_first(const GroupView &gv, uint32_t c, uint32_t off, uint2 *row)
{
    const uint32_t s4 = lane_id() & 3u;
    for (uint32_t e = s4; e < c; e += 4)
        row[e] = __ldcs(&gv.ent[off + e]);
    __syncwarp();
    M first = 0;
    for (uint32_t e = s4; e < c; e += 4) {
        const uint2 me = row[e];
        bool is = true;
        for (uint32_t j = 0; j < c; ++j) {
            const uint2 o = row[j];
            is = is && !(o.x == me.x && o.y < me.y);
        }
        first |= (M)is << e;
    }
    return group_or(first);
}

} // namespace mk
