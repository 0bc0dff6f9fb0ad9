// Incremental / decremental single-source shortest paths and BFS (paper,
// Algorithm "SSSP - Incremental / Decremental" and Sec. "Dynamic Single
// Source Shortest Path and Breadth First Search").
//
// Every vertex holds a 64-bit tree node <distance:32, parent:32>, updated
// with one 64-bit atomicMin so both halves change together (footnote on the
// tree-node packing); at the fixpoint the parent is the smallest-id tight
// predecessor.  Frontiers hold slab LISTS rather than edges or vertices: when
// a vertex improves, all its lists are enqueued (once per round, deduplicated
// by a per-vertex round stamp), and one warp then relaxes every live edge of
// one list.  Lists are short and evenly sized by the bucket rule, so the work
// is balanced even for high-degree vertices (the motivation of the paper's
// BucketIterator, Algorithm "Iteration Scheme 2").
//
// Decremental prologue: deleted tree edges (parent(v) = u) invalidate v; the
// invalidation then spreads to every tree descendant of such a v (the
// paper's per-vertex walk up the parent chain, done here as a union-find
// style find with path halving so that the walks share their work); then
// every edge from a valid vertex into an invalidated one is relaxed.  Incremental prologue: the edges inserted since
// the last commit, read with the UpdateIterator, are relaxed.  Common
// epilogue: rounds until no distance improves.
//
// The round loops run on the device: one persistent cooperative kernel
// executes all rounds of a phase and separates them with a grid barrier whose
// waits are bounded, so the host never reads a frontier size (the paper's
// host loop reads it every round).  If the cooperative launch is refused, the
// same round body runs as one launch per round driven by the host.
#include "mk_host.h"
#include "tma.cuh"
#include "walk.cuh"

#include <algorithm>

using namespace mk;

namespace {

constexpr uint32_t kInf32 = 0xFFFFFFFFu;
constexpr uint32_t kRoundsMaxThreads = 1024; // block size limit of the persistent round kernel
constexpr uint32_t kBarrierSpins = 1u << 24;

// consumer counter words (kConsumerWords)
enum {
    kCnt0 = 0,        // three rotating pairs <frontier size, blocks that have ended the round that filled it>
    kOverflow = 6,
    kInvTotal = 7,    // nonzero once this call invalidated a vertex
    kBar = 8,         // grid barrier: arrivals of the launch so far
    kFarCnt0 = 10,    // Near-Far ordering: sizes of the two far piles (10, 11),
    kClearWords = 12, // words [0, 12) are cleared at the start of every call
    kFarMin0 = 12,    // the smallest distance pushed to each pile (12, 13)
    kThresh = 14,     // the smallest source distance of the first frontier,
    kFarFirst0 = 15,  // and the round from which each pile is known to hold something (15, 16):
    kOrderWords = 5,  // words [12, 17) are set to INF by ordered calls
    kSoloR = 17,      // round index reached by a solo phase of block 0, and the frontier size there (18)
    kRoundsDone = 19,
    kRid = 20,        // last round stamp used (kept across calls)
    kPhase = 21       // Near-Far: last far-pile phase stamp used (kept across calls)
};

// The pair of frontier r, always accessed as one word: its size below 2^32,
// the blocks above.
__device__ __host__ __forceinline__ unsigned long long *count_of(uint32_t *ctr, uint32_t r)
{
    return reinterpret_cast<unsigned long long *>(ctr + kCnt0) + r % 3;
}

// A frontier of at most kSoloLists lists is processed by block 0 alone, with
// block-level barriers between rounds, for at most kSoloRounds rounds in a
// row (so the other blocks' bounded wait at the grid barrier never expires).
// Block 0 (one SM) has up to 192 four-lane groups: a frontier of up to
// about one list per group costs block 0 one load chain a round, less than
// a grid barrier plus one chain; a larger one is faster on the whole grid.
constexpr uint32_t kSoloLists = 192;
constexpr uint32_t kSoloRounds = 4096;
// A frontier of at most kDirectLists lists issues the atomic minima without
// reading the nodes first: a round trip less, and such rounds are made of round
// trips.  So does one of up to kDirectMost lists that is not much smaller than
// the one before: where each list goes on improving about another (a road
// grid: 3.78 -> 3.35 ms of rounds a pass), few of the minima are in vain; a
// frontier that shrinks is running out of improvements (R-MAT scale 20:
// everything up to 2^18 lists direct cost 9 % of the rounds).
constexpr uint32_t kDirectLists = 16384, kDirectMost = 1u << 18;
// Near-Far ordering: the far pile is split into the frontier whenever the
// frontier holds fewer lists than this (a smaller frontier costs a round
// about as much as a larger one).
constexpr uint32_t kNearMin = 2048;

__device__ __forceinline__ uint32_t node_dist(unsigned long long d) { return (uint32_t)(d >> 32); }
__device__ __forceinline__ uint32_t node_parent(unsigned long long d) { return (uint32_t)d; }

template <typename T>
__device__ __forceinline__ uint32_t ld_volatile(const T *p)
{
    return (uint32_t)*(volatile const T *)p;
}

} // namespace

// Arguments of the round loops (one struct so the cooperative launch passes
// a single pointer).
struct RoundArgs {
    GView g;
    unsigned long long *D;
    uint2 *front[2];      // list frontiers: <list, source of the list>
    uint32_t *ctr;        // consumer counter words
    uint32_t *stamp;
    uint32_t *inv;
    uint32_t cap;
    uint32_t max_hops;
    uint32_t max_rounds;
    uint32_t barrier_spins; // polls before a grid-barrier wait gives up
    uint32_t source;
    int unit;
    uint32_t *dist;       // the caller's outputs (nullable), written when the phase ends
    uint32_t *parent;
    uint32_t delta;       // Near-Far bucket width (0: plain frontier rounds)
    uint32_t *far[2];     // Near-Far: the two far piles (V vertices each)
    uint32_t *fstamp;     // Near-Far: phase in which a vertex last joined a pile
};

namespace {

// Near-Far ordering of the rounds (an addition to the paper's frontier
// rounds, for graphs of large diameter and weight range): an improvement
// to a distance at or above the split distance T does not enqueue the
// vertex's lists; the vertex joins the far pile instead (once per phase,
// through its pile stamp), and whenever the frontier is small the pile is
// split at a larger T.  Only the order of the relaxations changes: the rounds
// still run until no distance improves, so the result is the same fixpoint.
struct NearFar {
    uint32_t T = kInf32;      // split distance of this phase
    uint32_t phase = 0;       // pile stamp of this phase
    uint32_t *pile = nullptr; // the pile this phase appends to
    uint32_t *count = nullptr;
    uint32_t *dmin = nullptr; // smallest distance pushed to it
    // Smallest r such that a step before round r pushed to it.  Whether a pile
    // is split or a round run decides which barrier a block waits at next, so
    // every block has to decide alike; a block that runs round r ahead of the
    // others raises the pile's count, but can only set r + 1 here.
    uint32_t *first = nullptr;
};

// The pile of index k.
__device__ __forceinline__ NearFar far_pile(const RoundArgs &a, uint32_t k, uint32_t T, uint32_t phase)
{
    return {T, phase, a.far[k], a.ctr + kFarCnt0 + k, a.ctr + kFarMin0 + k, a.ctr + kFarFirst0 + k};
}

// A block's staging area for the far pile, as FrontierSmem for the frontier.
struct FarSmem {
    uint32_t buf[kRoundsMaxThreads / 32][kWarpBuf];
    uint32_t held[kRoundsMaxThreads / 32], at[kRoundsMaxThreads / 32];
    uint32_t dmin; // smallest distance pushed since the last flush
};

__device__ __forceinline__ void far_put(const RoundArgs &a, const NearFar &nf, uint32_t at, uint32_t y)
{
    if (at < a.g.V)
        nf.pile[at] = y;
    else
        *(int *)(a.ctr + kOverflow) = 1;
}

// Appends the lane's vertices y[k] with push[k] (distances d[k]) to the far
// pile, each once per phase: st[k] is the pile stamp that the caller exchanged
// for the phase's.  Must be called by the full warp.
template <int N>
__device__ __forceinline__ void far_push(const RoundArgs &a, const NearFar &nf, FarSmem &sm, const uint32_t (&y)[N],
                                         const bool (&push)[N], const uint32_t (&d)[N], const uint32_t (&stamps)[N])
{
    const uint32_t lane = lane_id(), w = threadIdx.x >> 5;
    bool any = false;
#pragma unroll
    for (int k = 0; k < N; ++k)
        any = any || push[k];
    if (!__any_sync(kFull, any))
        return;
    uint32_t st[N], c = 0, dm = kInf32;
#pragma unroll
    for (int k = 0; k < N; ++k)
        st[k] = push[k] ? stamps[k] : nf.phase;
#pragma unroll
    for (int k = 0; k < N; ++k)
        if (st[k] != nf.phase) {
            ++c;
            dm = min(dm, d[k]);
        } else if (push[k]) {
            dm = min(dm, d[k]); // in the pile already, at a larger distance
        }
    uint32_t incl = c;
#pragma unroll
    for (uint32_t o = 1; o < 32; o <<= 1) {
        const uint32_t t = __shfl_up_sync(kFull, incl, o);
        if (lane >= o)
            incl += t;
    }
    dm = __reduce_min_sync(kFull, dm);
    const uint32_t total = __shfl_sync(kFull, incl, 31), held = sm.held[w];
    const bool fits = held + total <= kWarpBuf;
    uint32_t base = 0;
    if (lane == 0)
        atomicMin(&sm.dmin, dm);
    if (!fits) {
        if (lane == 0)
            base = atomicAdd(nf.count, held + total);
        base = __shfl_sync(kFull, base, 0);
        for (uint32_t t = lane; t < held; t += 32)
            far_put(a, nf, base + t, sm.buf[w][t]);
    }
    uint32_t t = held + incl - c;
#pragma unroll
    for (int k = 0; k < N; ++k)
        if (st[k] != nf.phase) {
            if (fits)
                sm.buf[w][t] = y[k];
            else
                far_put(a, nf, base + t, y[k]);
            ++t;
        }
    __syncwarp();
    if (lane == 0)
        sm.held[w] = fits ? held + total : 0u;
    __syncwarp();
}

// Reserves the staged vertices' places in the pile: by one warp, between two
// barriers of the block (beside the frontier's reservation, so that a round
// waits for one of them only).  `round`: the first round after this step.
__device__ __forceinline__ void far_reserve(const NearFar &nf, FarSmem &sm, uint32_t round)
{
    constexpr uint32_t kWarps = kRoundsMaxThreads / 32;
    const uint32_t lane = lane_id();
    const uint32_t h = lane < kWarps ? sm.held[lane] : 0u;
    uint32_t incl = h;
#pragma unroll
    for (uint32_t o = 1; o < 32; o <<= 1) {
        const uint32_t t = __shfl_up_sync(kFull, incl, o);
        if (lane >= o)
            incl += t;
    }
    uint32_t base = 0;
    if (lane == 31) {
        if (sm.dmin != kInf32) { // something was pushed, staged still or not
            atomicMin(nf.dmin, sm.dmin);
            atomicMin(nf.first, round);
        }
        sm.dmin = kInf32;
        if (incl)
            base = atomicAdd(nf.count, incl);
    }
    base = __shfl_sync(kFull, base, 31);
    if (lane < kWarps)
        sm.at[lane] = base + incl - h;
}

// Then copies them, each warp its own; the caller synchronises the block
// before more are staged.
__device__ __forceinline__ void far_copy(const RoundArgs &a, const NearFar &nf, FarSmem &sm)
{
    const uint32_t lane = lane_id(), w = threadIdx.x >> 5;
    const uint32_t held = sm.held[w], at = sm.at[w];
    for (uint32_t t = lane; t < held; t += 32)
        far_put(a, nf, at + t, sm.buf[w][t]);
    __syncwarp();
    if (lane == 0)
        sm.held[w] = 0;
}

// Relaxes the lane's four edges (x, y[k], w[k]) with live[k] and enqueues
// the lists of each vertex whose distance this lane lowered first in this
// round (staged in the warp's frontier buffer).  The accesses of the four
// edges go out together, step by step: the four targets' tree nodes are
// read, then the atomic minima of the candidates that beat them are issued,
// then the improved targets' vinfo entries are read and their round stamps
// exchanged, so a slab costs three memory round trips per lane instead of
// three per edge.  A candidate that only names a smaller parent at the same
// distance changes the node but enqueues nothing: what leaves the vertex
// depends on its distance alone.  `direct` leaves the read of the nodes out
// and issues every minimum: one round trip less, more atomics, for the rounds
// whose time is their round trips.  Must be called by the full warp.
template <bool kNF = false, uint32_t kWarps, typename C>
__device__ __forceinline__ void relax_edges4(const RoundArgs &a, uint32_t x, uint32_t dx, const uint32_t (&y)[4],
                                             const uint32_t (&w)[4], const bool (&live)[4], uint32_t round,
                                             FrontierSmem<kWarps> &bq, uint2 *Fn, C *cnt, int *overflow,
                                             uint32_t &edges, uint32_t &improved,
                                             const NearFar *nf = nullptr, FarSmem *fs = nullptr,
                                             bool direct = false)
{
    // candidate of edge k: <nd[k], x>
    auto cand = [&](uint32_t d) { return ((unsigned long long)d << 32) | x; };
    uint32_t nd[4];
    unsigned long long cur[4];
    bool up[4];
    uint32_t n_live = 0;
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        n_live += live[k];
        const unsigned long long d = (unsigned long long)dx + (a.unit ? 1u : w[k]);
        up[k] = live[k] && d < kInf32;
        nd[k] = (uint32_t)d;
    }
    edges += n_live;
    if (direct) {
#pragma unroll
        for (int k = 0; k < 4; ++k)
            cur[k] = up[k] ? atomicMin(&a.D[y[k]], cand(nd[k])) : 0ull;
    } else {
#pragma unroll
        for (int k = 0; k < 4; ++k)
            cur[k] = up[k] ? __ldcg(&a.D[y[k]]) : 0ull;
#pragma unroll
        for (int k = 0; k < 4; ++k)
            if (up[k] && cand(nd[k]) < cur[k])
                cur[k] = atomicMin(&a.D[y[k]], cand(nd[k]));
            else
                up[k] = false;
    }
    bool any = false;
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        up[k] = up[k] && nd[k] < node_dist(cur[k]);
        any = any || up[k];
    }
    if (!__any_sync(kFull, any))
        return;
    // improvements at or beyond the split distance wait in the far pile
    bool fp[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        fp[k] = kNF && up[k] && nd[k] >= nf->T;
        up[k] = up[k] && !fp[k];
    }
    uint2 vi[4];
    uint32_t st[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        vi[k] = make_uint2(0, 0);
        st[k] = round;
        if (up[k])
            vi[k] = a.g.vinfo[y[k]];
        if (up[k] || (kNF && fp[k])) // one exchange, of the stamp that counts
            st[k] = atomicExch(kNF && fp[k] ? &a.fstamp[y[k]] : &a.stamp[y[k]], kNF && fp[k] ? nf->phase : round);
    }
    if (kNF)
        far_push<4>(a, *nf, *fs, y, fp, nd, st);
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        up[k] = up[k] && st[k] != round;
        improved += up[k];
    }
    enqueue_lists<4>(bq, y, up, vi, Fn, cnt, a.cap, overflow);
}

__device__ __forceinline__ unsigned long long warp_sum(unsigned long long v)
{
#pragma unroll
    for (int o = 16; o; o >>= 1)
        v += __shfl_xor_sync(kFull, v, o);
    return v;
}

// One round over frontier F[0, n): every 4-lane group of every warp takes
// one list at a time (group index + k * groups in the grid; eight lists per
// warp in flight), so a round's lists are spread over all warps; each
// group's entry, source distance and head slab are loaded one step ahead
// (the entry two steps ahead) while the current list is relaxed.  A frontier
// of at most `most` lists issues its minima directly (relax_edges4).
template <bool kNF = false, uint32_t kWarps, typename C>
__device__ __forceinline__ void relax_body(const RoundArgs &a, const uint2 *F, uint32_t n, uint2 *Fn, C *cnt,
                                           uint32_t round, uint32_t warp0, uint32_t nwarps, uint32_t most, FrontierSmem<kWarps> &bq,
                                           const NearFar *nf = nullptr, FarSmem *fs = nullptr)
{
    const GView &g = a.g;
    const bool direct = n <= most;
    const uint32_t s4 = lane_id() & 3u, g4 = lane_id() >> 2;
    int *overflow = (int *)(a.ctr + kOverflow);
    uint32_t lists = 0, slabs = 0, edges = 0, improved = 0;
    const uint32_t gs = nwarps * 8; // groups in the grid (indexes stay below H + 2 gs, far from 2^32)
    const uint2 none = make_uint2(kNil, 0);
    uint32_t i = warp0 * 8 + g4;
    // pipeline: entry e with its distance dx and head slab (lo, hi) (this
    // step), entry ne (next step)
    uint2 e = i < n ? __ldcg(&F[i]) : none;
    uint2 ne = i + gs < n ? __ldcg(&F[i + gs]) : none;
    uint32_t dx = e.x != kNil ? node_dist(__ldcg(&a.D[e.y])) : kInf32;
    uint4 lo, hi;
    group4_load(g, e.x, lo, hi);
    for (uint32_t base = warp0 * 8; base < n; base += gs, i += gs) {
        const uint2 nne = i + 2 * gs < n ? __ldcg(&F[i + 2 * gs]) : none;
        const uint32_t ndx = ne.x != kNil ? node_dist(__ldcg(&a.D[ne.y])) : kInf32;
        uint4 nlo, nhi;
        group4_load(g, ne.x, nlo, nhi);
        lists += __popc(__ballot_sync(kFull, e.x != kNil && s4 == 0));
        const uint32_t L = dx != kInf32 ? e.x : kNil;
        const uint32_t x = e.y, d = dx;
        slabs += walk_lists_g4_from(g, L, true, lo, hi, 0, a.max_hops,
                                    [&](const uint32_t(&y)[4], const uint32_t(&w)[4], const bool(&live)[4]) {
                                        relax_edges4<kNF>(a, x, d, y, w, live, round, bq, Fn, cnt, overflow,
                                                          edges, improved, nf, fs, direct);
                                    });
        e = ne;
        ne = nne;
        dx = ndx;
        lo = nlo;
        hi = nhi;
    }
    if (warp0 * 8 >= n)
        return;
    count_add(g.st, kCtrRelaxLists, lists);
    count_add(g.st, kCtrRelaxSlabs, slabs);
    count_add(g.st, kCtrRelaxEdges, warp_sum(edges));
    count_add(g.st, kCtrRelaxImproved, warp_sum(improved));
}

// Round r of a phase: relaxes frontier r (front[r & 1], n entries) and
// appends to frontier r + 1, whose size is counted in *cnt (a global counter
// or, in a solo phase, block 0's own).  Called by whole blocks: the block's
// staged entries are flushed at the end.
template <bool kNF = false, uint32_t kWarps, typename C>
__device__ __forceinline__ void round_step(const RoundArgs &a, C *cnt, uint32_t r, uint32_t n, uint64_t warp0,
                                           uint64_t nwarps, uint32_t rid, uint32_t most, FrontierSmem<kWarps> &bq,
                                           const NearFar *nf = nullptr, FarSmem *fs = nullptr)
{
    const uint32_t in = r & 1;
    relax_body<kNF>(a, a.front[in], n, a.front[in ^ 1], cnt, rid + 2 + r, warp0, nwarps, most, bq, nf, fs);
    frontier_flush(bq, a.front[in ^ 1], cnt, a.cap, (int *)(a.ctr + kOverflow), [&]() {
        if (kNF)
            far_reserve(*nf, *fs, r + 1);
    });
    if (kNF)
        far_copy(a, *nf, *fs);
}

__device__ __forceinline__ void fence_gpu() { asm volatile("fence.acq_rel.gpu;" ::: "memory"); }

__device__ __forceinline__ unsigned long long ld_acquire(const unsigned long long *p)
{
    unsigned long long v;
    asm volatile("ld.acquire.gpu.u64 %0, [%1];" : "=l"(v) : "l"(p) : "memory");
    return v;
}

// Ends the round that filled frontier r: waits until every block of the
// (cooperative) grid has, and returns the frontier's size in *n.  The blocks
// arrive in the high word of the pair whose low word counts the frontier, so
// the load that sees the last arrival brings the size with it.  Returns false
// when the wait gave up.  Called by whole blocks.
__device__ __forceinline__ bool round_barrier(uint32_t *ctr, uint32_t r, uint32_t max_spins, uint32_t *n)
{
    __shared__ uint32_t s_n, s_ok;
    __syncthreads();
    if (threadIdx.x == 0) {
        unsigned long long *pair = count_of(ctr, r);
        fence_gpu();
        atomicAdd(pair, 1ull << 32);
        uint32_t ok = 1, spins = 0;
        unsigned long long v = ld_acquire(pair);
        while ((uint32_t)(v >> 32) < gridDim.x) {
            if (++spins > max_spins) {
                ok = 0;
                break;
            }
            __nanosleep(20);
            v = ld_acquire(pair);
        }
        fence_gpu();
        s_n = (uint32_t)v;
        s_ok = ok;
    }
    __syncthreads();
    *n = s_n;
    return s_ok != 0;
}

// Bounded grid barrier for a co-resident (cooperative) grid on one counter
// that only grows: barrier k of a launch is passed once the counter reaches
// k * gridDim.x, so a block arrives with one atomicAdd and polls; nothing is
// reset between barriers (the counter is zeroed before each launch).
// `passed` is the block's count of barriers so far (thread 0's copy is the
// one used).  Returns false when the wait gave up.
__device__ bool grid_barrier(uint32_t *bar, uint32_t &passed, uint32_t max_spins)
{
    __shared__ int ok_s;
    __syncthreads();
    if (threadIdx.x == 0) {
        const uint32_t target = (++passed) * gridDim.x;
        fence_gpu();
        atomicAdd(bar, 1u);
        int ok = 1;
        uint32_t spins = 0;
        while ((int)(ld_volatile(bar) - target) < 0) {
            if (++spins > max_spins) {
                ok = 0;
                break;
            }
            __nanosleep(32);
        }
        fence_gpu();
        ok_s = ok;
    }
    __syncthreads();
    return ok_s != 0;
}

// Splits the far pile pile[0, fc) at T2 before round r: a vertex whose
// distance is now below T2 has its lists appended to frontier r (under the
// stamp of the entries already there, rid + 1 + r, so a vertex queued
// there already is not queued twice), every other one moves to the pile of
// `next` under its phase stamp.  Called by every thread of every block.
__device__ __forceinline__ void far_split(const RoundArgs &a, const uint32_t *pile, uint32_t fc, const NearFar &next,
                                          uint32_t T2, uint32_t r, uint32_t rid, uint64_t warp0, uint64_t nwarps,
                                          FrontierSmem<kRoundsMaxThreads / 32> &bq, FarSmem &fs)
{
    uint2 *out = a.front[r & 1];
    unsigned long long *cnt = count_of(a.ctr, r);
    const uint32_t stampv = rid + 1 + r;
    int *overflow = (int *)(a.ctr + kOverflow);
    for (uint64_t wb = warp0 * 32; wb < fc; wb += nwarps * 32) {
        const uint64_t i = wb + lane_id();
        const bool valid = i < fc;
        uint32_t y = 0, dy = kInf32;
        if (valid) {
            y = __ldcg(&pile[i]);
            dy = node_dist(__ldcg(&a.D[y]));
        }
        bool near = valid && dy < T2;
        uint2 vi = make_uint2(0, 0);
        uint32_t st = stampv;
        const bool far = valid && dy >= T2;
        if (near)
            vi = a.g.vinfo[y];
        if (valid)
            st = atomicExch(far ? &a.fstamp[y] : &a.stamp[y], far ? next.phase : stampv);
        const uint32_t ys[1] = {y};
        const bool ups[1] = {near && st != stampv};
        const uint2 vis[1] = {vi};
        enqueue_lists<1>(bq, ys, ups, vis, out, cnt, a.cap, overflow);
        const bool fars[1] = {far};
        const uint32_t ds[1] = {dy}, sts[1] = {st};
        far_push<1>(a, next, fs, ys, fars, ds, sts);
    }
    frontier_flush(bq, out, cnt, a.cap, overflow, [&]() { far_reserve(next, fs, r); });
    far_copy(a, next, fs);
}

} // namespace

// All rounds of one phase in one cooperative launch.  The phase input is
// front[0] with its size in ctr[kCnt0]; the rotating pairs must be zero.  Large
// frontiers are processed by the whole grid, one grid barrier per round.
// While the frontier stays small, block 0 runs the rounds alone (its warps
// striding over the frontier, its frontier sizes in shared memory,
// __syncthreads between rounds) for at most kSoloRounds rounds; the solo
// phase sits between two grid barriers, so no block reads a global size
// while block 0 changes them, and the others wait at one barrier instead of
// one per round.
//
// A round is bound by its chain of dependent accesses (frontier entry, slab
// and source node, target nodes, atomic minimum, index and stamp): 3.5-5 us
// for up to one list a group, then 2.3 us for the flush, the barrier and the
// next size (7.3 us in all, 9.5 before the size came with the barrier, the
// warps were spread over the SMs and small rounds went without the nodes'
// read).  A large round runs at 7-12 G lists/s; what held it was the frontier
// count, on which every append past a block's buffer met.  R-MAT scale 20
// from the hub: BFS 540 -> 266 us, SSSP 990 -> 510 us.
template <bool kNF>
__global__ void __launch_bounds__(kRoundsMaxThreads, 1) k_rounds(RoundArgs a)
{
    __shared__ uint32_t solo_cnt[3];
    __shared__ FrontierSmem<kRoundsMaxThreads / 32> bq;
    __shared__ FarSmem fs[1];
    __shared__ uint32_t s_word, s_fc, s_fm, s_first;
    if (threadIdx.x == 0)
        s_word = ld_volatile(count_of(a.ctr, 0));
    if (kNF) {
        if (threadIdx.x < kRoundsMaxThreads / 32)
            fs[0].held[threadIdx.x] = 0;
        if (threadIdx.x == 0)
            fs[0].dmin = kInf32;
    }
    frontier_init(bq);
    // consecutive warps of the frontier sit on different SMs, so that a
    // frontier of a few thousand lists is relaxed by all of them
    const uint64_t warp0 = (uint64_t)(threadIdx.x >> 5) * gridDim.x + blockIdx.x;
    const uint64_t nwarps = ((uint64_t)gridDim.x * blockDim.x) >> 5;
    const uint32_t rid = __ldg(a.ctr + kRid);
    uint32_t r = 0, bars = 0, passed = 0;
    uint32_t before = 0; // lists of the last round of the whole grid, none after other steps
    bool ok = true;
    // a frontier never holds more than `cap` entries; a larger count
    // (entries dropped on overflow, reported below) is read as cap
    uint32_t n = min(s_word, a.cap);
    // Near-Far: the first split distance is delta above the smallest source
    // distance of the first frontier (ctr[kThresh] starts at INF)
    NearFar nf;
    uint32_t cur = 0, splits = 0, burst = 0;
    const uint32_t phase0 = kNF ? __ldg(a.ctr + kPhase) + 1 : 0;
    if (kNF) {
        uint32_t m = kInf32;
        for (uint64_t i = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; i < n;
             i += (uint64_t)gridDim.x * blockDim.x)
            m = min(m, node_dist(__ldcg(&a.D[__ldcg(&a.front[0][i].y)])));
        m = __reduce_min_sync(kFull, m);
        if ((threadIdx.x & 31) == 0 && m != kInf32)
            atomicMin(a.ctr + kThresh, m);
        ++bars;
        ok = grid_barrier(a.ctr + kBar, passed, a.barrier_spins);
        const uint32_t t0 = ld_volatile(a.ctr + kThresh);
        nf = far_pile(a, 0, t0 >= kInf32 - a.delta ? kInf32 : t0 + a.delta, phase0);
    }
    while (ok && r < a.max_rounds) {
        if (kNF && n < kNearMin) {
            // one read of the pile's words per block; its size and smallest
            // distance are final where `first` says that it is split
            if (threadIdx.x == 0) {
                s_first = ld_volatile(a.ctr + kFarFirst0 + cur);
                s_fc = ld_volatile(a.ctr + kFarCnt0 + cur);
                s_fm = ld_volatile(a.ctr + kFarMin0 + cur);
            }
            __syncthreads();
            const uint32_t fc = min(s_fc, a.g.V), fm = s_fm;
            if (s_first <= r) {
                // the near frontier is small: move the far pile's vertices
                // below the next split distance into it, once every block
                // has read the words above; the distance grows with each
                // split in a row
                ++bars;
                if (!grid_barrier(a.ctr + kBar, passed, a.barrier_spins)) {
                    ok = false;
                    break;
                }
                const uint32_t base = max(nf.T, fm);
                const uint64_t width = (uint64_t)a.delta << min(burst, 16u);
                ++splits;
                const NearFar next = far_pile(a, cur ^ 1, (uint64_t)base + width >= kInf32 ? kInf32 : (uint32_t)(base + width),
                                              phase0 + splits);
                far_split(a, nf.pile, fc, next, next.T, r, rid, warp0, nwarps, bq, fs[0]);
                ++bars;
                if (!grid_barrier(a.ctr + kBar, passed, a.barrier_spins)) {
                    ok = false;
                    break;
                }
                // the old pile is empty again; no block reads its words
                // before the next split, two grid barriers on
                if (threadIdx.x == 0) {
                    if (blockIdx.x == 0) {
                        a.ctr[kFarCnt0 + cur] = 0;
                        a.ctr[kFarMin0 + cur] = kInf32;
                        a.ctr[kFarFirst0 + cur] = kInf32;
                    }
                    s_word = ld_volatile(count_of(a.ctr, r));
                }
                __syncthreads();
                n = min(s_word, a.cap);
                cur ^= 1;
                nf = next;
                ++burst;
                if (splits > a.max_rounds) {
                    ok = false;
                    break;
                }
                continue;
            }
        }
        burst = 0;
        if (n == 0)
            break;
        if (n > kSoloLists) {
            // the pair of frontier r - 1, which every block has left, is
            // that of frontier r + 2
            if (blockIdx.x == 0 && threadIdx.x == 0)
                *count_of(a.ctr, r + 2) = 0;
            const uint32_t most = before && n >= before - before / 4 ? kDirectMost : kDirectLists;
            before = n;
            round_step<kNF>(a, count_of(a.ctr, r + 1), r, n, warp0, nwarps, rid, most, bq, &nf, fs);
            ++bars;
            ++r;
            ok = round_barrier(a.ctr, r, a.barrier_spins, &n);
            n = min(n, a.cap);
            continue;
        }
        // every block has read n: block 0 may now change the global sizes
        bars += 2;
        if (!grid_barrier(a.ctr + kBar, passed, a.barrier_spins)) {
            ok = false;
            break;
        }
        if (blockIdx.x == 0) {
            const uint64_t bw0 = threadIdx.x >> 5, bnw = blockDim.x >> 5;
            if (threadIdx.x < 3)
                solo_cnt[threadIdx.x] = 0;
            __syncthreads();
            uint32_t steps = 0;
            do {
                round_step<kNF>(a, &solo_cnt[(r + 1) % 3], r, n, bw0, bnw, rid, kDirectLists, bq, &nf, fs);
                __syncthreads();
                ++r;
                ++steps;
                n = min(*(volatile uint32_t *)&solo_cnt[r % 3], a.cap);
                // written again two rounds on
                if (threadIdx.x == 0)
                    solo_cnt[(r + 2) % 3] = 0;
            } while (n > 0 && n <= kSoloLists && steps < kSoloRounds && r < a.max_rounds);
            if (threadIdx.x == 0) {
                *count_of(a.ctr, r) = n;
                for (uint32_t k = 1; k < 3; ++k)
                    *count_of(a.ctr, r + k) = 0;
                a.ctr[kSoloR] = r;
                a.ctr[kSoloR + 1] = n;
            }
        }
        if (!grid_barrier(a.ctr + kBar, passed, a.barrier_spins)) {
            ok = false;
            break;
        }
        if (threadIdx.x == 0) {
            s_word = ld_volatile(a.ctr + kSoloR);
            s_fc = ld_volatile(a.ctr + kSoloR + 1);
        }
        __syncthreads();
        r = s_word;
        n = s_fc;
        before = 0;
        __syncthreads(); // every thread has read them before thread 0 rewrites them
    }
    // The phase is over: every block left the loop at the same round, after
    // the grid barrier that ended the last relaxation, so D is final.  The
    // call's epilogue runs here instead of in two more launches: the tree
    // nodes go to the caller's arrays, and the round stamp moves past every
    // id this call used.
    if (a.dist || a.parent) {
        const uint64_t stride = (uint64_t)gridDim.x * blockDim.x;
        for (uint64_t v = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; v < a.g.V; v += stride) {
            const unsigned long long d = __ldcg(&a.D[v]);
            if (a.dist)
                a.dist[v] = node_dist(d);
            if (a.parent)
                a.parent[v] = node_parent(d);
        }
    }
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        a.ctr[kRoundsDone] = r;
        a.ctr[kRid] += r + 2;
        if (kNF)
            a.ctr[kPhase] = phase0 + splits;
        atomicAdd(&a.g.st->ctr[kCtrRounds][0], (unsigned long long)r);
        atomicAdd(&a.g.st->ctr[kCtrGridBarriers][0], (unsigned long long)bars);
        if (a.dist || a.parent)
            atomicAdd(&a.g.st->ctr[kCtrUnpacked][0], (unsigned long long)a.g.V);
        if (!ok || r >= a.max_rounds || ld_volatile(a.ctr + kOverflow) != 0)
            set_status(a.g.st, kErrTimeout);
    }
}

// One round, for the host-driven fallback.
__global__ void __launch_bounds__(256) k_round_once(RoundArgs a, uint32_t r, uint32_t n)
{
    __shared__ FrontierSmem<8> bq;
    frontier_init(bq);
    const uint64_t warp0 = (blockIdx.x * (uint64_t)blockDim.x + threadIdx.x) >> 5;
    const uint64_t nwarps = ((uint64_t)gridDim.x * blockDim.x) >> 5;
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        *count_of(a.ctr, r + 2) = 0;
        a.ctr[kRoundsDone] = r + 1;
    }
    round_step(a, count_of(a.ctr, r + 1), r, n, warp0, nwarps, __ldg(a.ctr + kRid), kDirectLists, bq);
}

__global__ void k_sssp_init(unsigned long long *D, uint32_t V, uint32_t source, uint2 *front, uint32_t *count,
                            const uint2 *vinfo)
{
    const uint32_t v = blockIdx.x * blockDim.x + threadIdx.x;
    if (v < V)
        D[v] = v == source ? ((unsigned long long)0 << 32 | source) : kInfNode;
    if (v == 0) {
        const uint2 vi = vinfo[source];
        for (uint32_t b = 0; b < vi.y; ++b)
            front[b] = make_uint2(vi.x + b, source);
        *count = vi.y;
    }
}

// Decremental seeds: a deleted edge (u, v) that is v's tree edge invalidates
// v (its tree node becomes <INF, INVALID> and its bit is set in `inv`).
__global__ void k_invalidate(const unsigned long long *dlog, uint64_t n, RoundArgs a)
{
    const uint64_t i = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x;
    bool hit = false;
    uint32_t v = 0;
    const unsigned long long e = i < n ? __ldcs(&dlog[i]) : ~0ull; // all-ones: nothing was removed
    if (e != ~0ull) {
        const uint32_t u = (uint32_t)(e >> 32);
        v = (uint32_t)e;
        const unsigned long long dv = __ldcg(&a.D[v]);
        hit = v != a.source && dv != kInfNode && node_parent(dv) == u && atomicCAS(&a.D[v], dv, kInfNode) == dv;
    }
    if (hit)
        atomicOr(&a.inv[v >> 5], 1u << (v & 31));
    const uint32_t m = __ballot_sync(kFull, hit);
    if (m && lane_id() == 0)
        a.ctr[kInvTotal] = 1; // a flag: something was invalidated
    count_add(a.g.st, kCtrInvalidated, __popc(m));
}

// The invalidation spreads to every tree descendant of the seeds: a vertex
// is invalid iff the path from it up the shortest-path tree reaches a seed
// before the source.  As in the paper, each reached vertex walks its tree
// parents up until it meets the source (valid) or a vertex without a tree
// node (invalid: a seed, or a vertex this pass has already invalidated);
// invalid vertices get <INF, INVALID> at once, so later walks through them
// stop there.  Tree parents have strictly smaller distances (weights are
// >= 1), so every walk ends.  The loads are plain (L1-cacheable): the upper
// part of the tree, where most walks pass, stays in L1, and a stale line can
// only hide an invalidation made by this pass, whose walk went on up the
// same parents to the same seed, so the outcome is the same.  The
// invalidated vertices of one warp set their bits with one atomicOr (32
// consecutive vertices share a bitmap word).
__global__ void k_inv_walk(RoundArgs a)
{
    const uint32_t v = blockIdx.x * blockDim.x + threadIdx.x;
    if ((v & ~31u) >= a.g.V)
        return;
    count_add(a.g.st, kCtrWalkVertices, __popc(__ballot_sync(kFull, v < a.g.V)));
    bool bad = false;
    const unsigned long long dv = v < a.g.V && v != a.source ? a.D[v] : kInfNode;
    if (dv != kInfNode) {
        // only parents are read: a tree node's parent word is kNil exactly
        // when the node is <INF, INVALID> (every finite node names a
        // vertex), so one 4-byte load and one compare decide a hop; four
        // hops an iteration, the bound checked once per four
        const uint32_t *par = reinterpret_cast<const uint32_t *>(a.D); // low word of node x: par[2x]
        uint32_t x = node_parent(dv), hops = 0;
        while (x != a.source) {
            uint32_t p = par[2 * (uint64_t)x];
            if (p == kNil) {
                bad = true;
                break;
            }
            if (p == a.source)
                break;
            p = par[2 * (uint64_t)p];
            if (p == kNil) {
                bad = true;
                break;
            }
            if (p == a.source)
                break;
            p = par[2 * (uint64_t)p];
            if (p == kNil) {
                bad = true;
                break;
            }
            if (p == a.source)
                break;
            p = par[2 * (uint64_t)p];
            if (p == kNil) {
                bad = true;
                break;
            }
            x = p;
            if ((hops += 4) > a.max_rounds) { // parent pointers not a tree: corrupted state
                set_status(a.g.st, kErrTimeout);
                break;
            }
        }
    }
    if (bad)
        a.D[v] = kInfNode;
    const uint32_t mask = __ballot_sync(kFull, bad);
    if (lane_id() == 0 && mask) {
        atomicOr(&a.inv[v >> 5], mask);
        a.ctr[kInvTotal] = 1;
        count_add(a.g.st, kCtrInvalidated, __popc(mask));
    }
}

// After invalidation: relax every edge out of a valid vertex into a vertex
// invalidated by this call.  The target test reads the invalidation bitmap,
// which stays fixed during the pass, so every such edge is relaxed even after
// another in-neighbour has already given its target a finite distance; does
// nothing if nothing was invalidated.  A streaming scan over the whole slab
// array: a warp takes 32 consecutive slabs, reads their owners and the owners'
// tree nodes (two and one chunk ahead), and then the slabs whose source has a
// finite distance, eight lanes a slab, 16 bytes a lane.  Few edges lead to an
// invalidated vertex, so what bounds the pass is the reading and the tests:
// kBits 1 keeps the bitmap in shared memory, where a test is a word out of
// 32 banks instead of a line of L1 for each of a warp's keys; 2 reads it from
// memory where it does not fit.  Only distances change here (64-bit atomic
// minima whose results are not needed); the improved targets are enqueued by
// k_enqueue_invalid.  R-MAT scale 20: 122 us with bulk copies into shared
// memory, a lane a slab and the bitmap in L1, 77 us so (scale 17: 24 -> 16 us).
constexpr uint32_t kInvThreads = 1024;

template <int kBits>
__global__ void __launch_bounds__(kInvThreads, 1) k_relax_into_invalid_slabs(RoundArgs a)
{
    extern __shared__ uint32_t s_inv[];
    const GView &g = a.g;
    if (__ldg(a.ctr + kInvTotal) == 0) // set by the kernels before this one
        return;
    if (kBits == 1) {
        for (uint32_t i = threadIdx.x; i < (g.V + 31) / 32; i += kInvThreads)
            s_inv[i] = __ldg(&a.inv[i]);
        __syncthreads();
    }
    auto invalid = [&](uint32_t v) -> uint32_t {
        return ((kBits == 1 ? s_inv[v >> 5] : __ldg(&a.inv[v >> 5])) >> (v & 31u)) & 1u;
    };
    const uint32_t lane = lane_id(), gr = lane >> 3, sub = lane & 7u;
    const uint64_t total = (uint64_t)g.H + g.P, stride = (((uint64_t)gridDim.x * kInvThreads) >> 5) * 32;
    auto owner_of = [&](uint64_t c) { return c + lane < total ? __ldcg(&g.owner[c + lane]) : kNil; };
    auto dist_of = [&](uint32_t own) { return own != kNil ? node_dist(__ldcg(&a.D[own])) : kInf32; };
    // per-lane tallies, summed over the warp once at the end
    uint32_t slabs = 0, edges = 0, owners = 0, targets = 0;
    uint64_t c = ((blockIdx.x * (uint64_t)kInvThreads + threadIdx.x) >> 5) * 32;
    uint32_t own = owner_of(c), own1 = owner_of(c + stride), dx = dist_of(own);
    for (; c < total; c += stride) {
        const uint32_t live = __ballot_sync(kFull, dx != kInf32); // slabs of unreached or invalidated sources are not read
        uint4 part[8];
        const uint4 *at = reinterpret_cast<const uint4 *>(slab_ptr(g, (uint32_t)c + gr)) + sub;
#pragma unroll
        for (uint32_t j = 0; j < 8; ++j)
            part[j] = (live >> (4 * j + gr)) & 1u ? __ldcg(at + j * 32) : make_uint4(kEmptyKey, 0u, kEmptyKey, 0u);
        const uint32_t own2 = owner_of(c + 2 * stride), dx1 = dist_of(own1);
        owners += own != kNil;
        slabs += dx != kInf32;
#pragma unroll
        for (uint32_t j = 0; j < 8; ++j) {
            if (((live >> (4 * j)) & 15u) == 0)
                continue;
            const bool k0 = part[j].x < kTombKey, k1 = sub != 7u && part[j].z < kTombKey;
            edges += (k0 ? 1u : 0u) + (k1 ? 1u : 0u);
            const uint32_t h0 = k0 ? invalid(part[j].x) : 0u, h1 = k1 ? invalid(part[j].z) : 0u;
            if (!__any_sync(kFull, h0 | h1))
                continue;
            const uint32_t from = __shfl_sync(kFull, own, 4 * j + gr), d = __shfl_sync(kFull, dx, 4 * j + gr);
            targets += h0 + h1;
            const unsigned long long n0 = (unsigned long long)d + (a.unit ? 1u : part[j].y);
            const unsigned long long n1 = (unsigned long long)d + (a.unit ? 1u : part[j].w);
            if (h0 && n0 < kInf32)
                atomicMin(&a.D[part[j].x], (n0 << 32) | from);
            if (h1 && n1 < kInf32)
                atomicMin(&a.D[part[j].z], (n1 << 32) | from);
        }
        own = own1;
        own1 = own2;
        dx = dx1;
    }
    count_add(g.st, kCtrScanOwners, __reduce_add_sync(kFull, owners));
    count_add(g.st, kCtrScanSlabs, __reduce_add_sync(kFull, slabs));
    count_add(g.st, kCtrScanEdges, __reduce_add_sync(kFull, edges));
    count_add(g.st, kCtrScanTargets, __reduce_add_sync(kFull, targets));
}

// Enqueues the lists of every vertex invalidated by this call that the pass
// above gave a finite distance (one warp per 32-vertex word of the bitmap),
// stamped with the prologue's round so that the incremental prologue does
// not enqueue it again.  The frontier slots of vertices with few lists are
// reserved with one atomicAdd per block (a warp-level reservation would put
// one atomic per 32 vertices on the single frontier counter); a vertex with
// many lists is written by its whole warp.
__global__ void __launch_bounds__(256) k_enqueue_invalid(RoundArgs a)
{
    constexpr uint32_t kSmall = 8;
    __shared__ uint32_t s_total, s_base;
    const uint32_t lane = lane_id();
    const uint64_t word = (blockIdx.x * (uint64_t)blockDim.x + threadIdx.x) >> 5;
    if (threadIdx.x == 0)
        s_total = 0;
    __syncthreads();
    bool pred = false;
    uint2 vi = make_uint2(0, 0);
    const uint32_t y = (uint32_t)word * 32 + lane;
    if (word < ((uint64_t)a.g.V + 31) / 32 && __ldg(a.ctr + kInvTotal) != 0) {
        const uint32_t bits = __ldcg(&a.inv[word]);
        pred = (bits >> lane) & 1u;
        if (pred) {
            pred = __ldcg(&a.D[y]) != kInfNode;
            if (pred) {
                vi = a.g.vinfo[y];
                a.stamp[y] = __ldg(a.ctr + kRid) + 1;
            }
        }
    }
    count_add(a.g.st, kCtrScanImproved, __popc(__ballot_sync(kFull, pred)));
    // small vertices: warp scan of bucket counts, then a block reservation
    const bool small = pred && vi.y <= kSmall;
    const uint32_t c = small ? vi.y : 0;
    uint32_t incl = c;
#pragma unroll
    for (uint32_t o = 1; o < 32; o <<= 1) {
        const uint32_t t = __shfl_up_sync(kFull, incl, o);
        if (lane >= o)
            incl += t;
    }
    const uint32_t wtotal = __shfl_sync(kFull, incl, 31);
    uint32_t woff = 0;
    if (lane == 0 && wtotal)
        woff = atomicAdd(&s_total, wtotal);
    __syncthreads();
    if (threadIdx.x == 0 && s_total)
        s_base = atomicAdd(a.ctr + kCnt0, s_total);
    __syncthreads();
    int *overflow = (int *)(a.ctr + kOverflow);
    if (wtotal) {
        const uint32_t at = s_base + __shfl_sync(kFull, woff, 0) + incl - c;
        for (uint32_t k = 0; k < c; ++k) {
            if (at + k < a.cap)
                a.front[0][at + k] = make_uint2(vi.x + k, y);
            else
                *overflow = 1;
        }
    }
    // large vertices: one at a time, written by the whole warp
    uint32_t big = __ballot_sync(kFull, pred && !small);
    while (big) {
        const uint32_t l = __ffs(big) - 1;
        big &= big - 1;
        const uint32_t first = __shfl_sync(kFull, vi.x, l), nb = __shfl_sync(kFull, vi.y, l);
        const uint32_t yl = __shfl_sync(kFull, y, l);
        uint32_t base = 0;
        if (lane == 0)
            base = atomicAdd(a.ctr + kCnt0, nb);
        base = __shfl_sync(kFull, base, 0);
        for (uint32_t k = lane; k < nb; k += 32) {
            if (base + k < a.cap)
                a.front[0][base + k] = make_uint2(first + k, yl);
            else
                *overflow = 1;
        }
    }
}


// Incremental seeds: relax the entries inserted since the last commit.
// Every list in the updated-list log is walked from its UpdateIterator start
// (the marker slab, skipping its lanes before the marker lane, or all of it
// when it is full).  Every 4-lane group of every warp takes one list at a
// time (group index + k * groups in the grid; eight lists per warp in
// flight); the next list's log entry, source and marker are loaded a step
// ahead.
__global__ void __launch_bounds__(256, 5) k_relax_updated(RoundArgs a)
{
    const GView &g = a.g;
    const uint32_t s4 = lane_id() & 3u, g4 = lane_id() >> 2;
    const uint32_t n = min(__ldg(&g.st->ulog_count), g.H);
    const uint64_t warp0 = (blockIdx.x * (uint64_t)blockDim.x + threadIdx.x) >> 5;
    const uint64_t gs = (((uint64_t)gridDim.x * blockDim.x) >> 5) * 8; // 4-lane groups in the grid
    __shared__ FrontierSmem<8> bq;
    frontier_init(bq);
    const uint32_t round = __ldg(a.ctr + kRid) + 1;
    int *overflow = (int *)(a.ctr + kOverflow);
    uint32_t lists = 0, slabs = 0, edges = 0, improved = 0;
    uint64_t i = warp0 * 8 + g4;
    uint32_t L = i < n ? g.ulog[i] : kNil;
    uint32_t nL = i + gs < n ? g.ulog[i + gs] : kNil;
    uint32_t src = L != kNil ? g.list_src[L] : 0;
    unsigned long long mk = L != kNil ? g.lmark[L] : 0;
    for (uint64_t base = warp0 * 8; base < n; base += gs, i += gs) {
        const uint32_t nnL = i + 2 * gs < n ? g.ulog[i + 2 * gs] : kNil;
        const uint32_t nsrc = nL != kNil ? g.list_src[nL] : 0;
        const unsigned long long nmk = nL != kNil ? g.lmark[nL] : 0;
        const uint32_t dx = L != kNil ? node_dist(__ldcg(&a.D[src])) : kInf32;
        const uint32_t mlane = (uint32_t)(mk & 0xFF);
        const uint32_t first_lane = mlane == kInvalidLane ? 32u : mlane;
        const bool go = L != kNil && dx != kInf32;
        const uint32_t start = go ? (uint32_t)(mk >> 32) : kNil;
        uint4 lo, hi;
        group4_load(g, start, lo, hi);
        lists += __popc(__ballot_sync(kFull, go && s4 == 0));
        const uint32_t x = src;
        slabs += walk_lists_g4_from(g, start, true, lo, hi, first_lane, a.max_hops,
                                    [&](const uint32_t(&y)[4], const uint32_t(&w)[4], const bool(&live)[4]) {
                                        relax_edges4(a, x, dx, y, w, live, round, bq, a.front[0], a.ctr + kCnt0,
                                                     overflow, edges, improved);
                                    });
        L = nL;
        nL = nnL;
        src = nsrc;
        mk = nmk;
    }
    frontier_flush(bq, a.front[0], a.ctr + kCnt0, a.cap, overflow);
    count_add(g.st, kCtrSeedLists, lists);
    count_add(g.st, kCtrSeedSlabs, slabs);
    count_add(g.st, kCtrSeedEdges, warp_sum(edges));
    count_add(g.st, kCtrSeedImproved, warp_sum(improved));
}

// Incremental seeds from the inserted-edge log (the paper's incremental
// frontier is the batch's inserted edges), used when the epoch holds no
// deletes, so every logged edge is still live with its stored weight: each
// lane takes four consecutive log entries <src, dst, w> and relaxes them
// together, as relax_edges4 does a slab's four pairs (the sources' tree
// nodes, the targets' tree nodes, the atomic minima of the candidates that
// beat them, then the improved targets' vertex index entries and round
// stamps), and enqueues the lists of each vertex it lowered first in this
// round.  Two dependent gathers per edge instead of the walk's five loads
// per updated list (log entry, list source, marker, source node, slab).
__global__ void __launch_bounds__(256) k_relax_inserted(RoundArgs a, const uint4 *__restrict__ ilog, uint64_t n)
{
    __shared__ FrontierSmem<8> bq;
    frontier_init(bq);
    const uint32_t round = __ldg(a.ctr + kRid) + 1;
    int *overflow = (int *)(a.ctr + kOverflow);
    unsigned long long entries = 0, edges = 0, improved = 0;
    const uint64_t lane4 = (uint64_t)lane_id() * 4;
    const uint64_t stride = (uint64_t)gridDim.x * blockDim.x * 4;
    for (uint64_t wb = ((blockIdx.x * (uint64_t)blockDim.x + threadIdx.x) & ~31ull) * 4; wb < n; wb += stride) {
        uint32_t x[4], y[4], nd[4];
        bool up[4];
        unsigned long long cur[4];
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            const uint64_t i = wb + lane4 + k;
            const uint4 e = i < n ? __ldcs(&ilog[i]) : make_uint4(kNil, 0, 0, 0); // kNil: nothing was stored
            x[k] = e.x;
            y[k] = e.y;
            nd[k] = e.z;
            up[k] = e.x != kNil;
        }
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            entries += __popc(__ballot_sync(kFull, up[k]));
            const uint32_t dx = up[k] ? node_dist(__ldcg(&a.D[x[k]])) : kInf32;
            const unsigned long long d = (unsigned long long)dx + (a.unit ? 1u : nd[k]);
            up[k] = up[k] && dx != kInf32 && d < kInf32;
            nd[k] = (uint32_t)d;
        }
        auto cand = [&](int k) { return ((unsigned long long)nd[k] << 32) | x[k]; };
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            edges += __popc(__ballot_sync(kFull, up[k]));
            cur[k] = up[k] ? __ldcg(&a.D[y[k]]) : 0ull;
        }
#pragma unroll
        for (int k = 0; k < 4; ++k)
            if (up[k] && cand(k) < cur[k])
                cur[k] = atomicMin(&a.D[y[k]], cand(k));
            else
                up[k] = false;
        uint2 vi[4];
        uint32_t st[4];
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            up[k] = up[k] && nd[k] < node_dist(cur[k]);
            vi[k] = make_uint2(0, 0);
            st[k] = round;
            if (up[k]) {
                vi[k] = a.g.vinfo[y[k]];
                st[k] = atomicExch(&a.stamp[y[k]], round);
            }
        }
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            up[k] = up[k] && st[k] != round;
            improved += __popc(__ballot_sync(kFull, up[k]));
        }
        enqueue_lists<4>(bq, y, up, vi, a.front[0], a.ctr + kCnt0, a.cap, overflow);
    }
    frontier_flush(bq, a.front[0], a.ctr + kCnt0, a.cap, overflow);
    count_add(a.g.st, kCtrSeedLog, entries);
    count_add(a.g.st, kCtrSeedEdges, edges);
    count_add(a.g.st, kCtrSeedImproved, improved);
}

// Ends a call of the host-driven fallback (the round kernel does this
// itself): advances the round stamp past every id used (`rounds` rounds),
// reports an overflowed frontier.
__global__ void k_sssp_finish(uint32_t *ctr, DevState *st, uint32_t rounds)
{
    ctr[kRoundsDone] = rounds;
    ctr[kRid] += rounds + 2;
    if (ctr[kOverflow])
        set_status(st, kErrTimeout);
}

__global__ void k_unpack(const unsigned long long *D, uint32_t V, uint32_t *dist, uint32_t *parent)
{
    const uint32_t v = blockIdx.x * blockDim.x + threadIdx.x;
    if (v >= V)
        return;
    const unsigned long long d = D[v];
    if (dist)
        dist[v] = node_dist(d);
    if (parent)
        parent[v] = node_parent(d);
}

// ------------------------------------------------- several states, one pass
//
// mk_incr_multi advances up to kMaxMulti BFS/SSSP states of one graph
// together: the passes that read the graph's change log or its whole slab
// array (the incremental prologue over the updated lists, the decremental
// relax-into-invalid scan) and the round loop run once for all of them, each
// slab or list read once and relaxed into every state, the rounds of all
// states sharing one grid barrier per round.

constexpr uint32_t kMaxMulti = 4;

struct MultiArgs {
    RoundArgs c[kMaxMulti];
    uint32_t k; // states in use
};

// The incremental prologue (k_relax_updated) for every state at once: each
// logged list is walked once from its UpdateIterator start and every slab's
// new edges are relaxed into each state whose copy of the list's source has
// a finite distance.  Dynamic shared memory: one staging area per state.
__global__ void __launch_bounds__(256, 5) k_relax_updated_multi(MultiArgs m)
{
    extern __shared__ unsigned char multi_smem[];
    FrontierSmem<8> *bqs = reinterpret_cast<FrontierSmem<8> *>(multi_smem);
    const GView &g = m.c[0].g;
    const uint32_t s4 = lane_id() & 3u, g4 = lane_id() >> 2;
    const uint32_t n = min(__ldg(&g.st->ulog_count), g.H);
    const uint64_t warp0 = (blockIdx.x * (uint64_t)blockDim.x + threadIdx.x) >> 5;
    const uint64_t gs = (((uint64_t)gridDim.x * blockDim.x) >> 5) * 8;
    for (uint32_t j = 0; j < m.k; ++j)
        frontier_init(bqs[j]);
    uint32_t round[kMaxMulti];
#pragma unroll
    for (uint32_t j = 0; j < kMaxMulti; ++j)
        round[j] = j < m.k ? __ldg(m.c[j].ctr + kRid) + 1 : 0u;
    uint32_t lists = 0, slabs = 0, edges = 0, improved = 0;
    uint64_t i = warp0 * 8 + g4;
    uint32_t L = i < n ? g.ulog[i] : kNil;
    uint32_t nL = i + gs < n ? g.ulog[i + gs] : kNil;
    uint32_t src = L != kNil ? g.list_src[L] : 0;
    unsigned long long mk = L != kNil ? g.lmark[L] : 0;
    for (uint64_t base = warp0 * 8; base < n; base += gs, i += gs) {
        const uint32_t nnL = i + 2 * gs < n ? g.ulog[i + 2 * gs] : kNil;
        const uint32_t nsrc = nL != kNil ? g.list_src[nL] : 0;
        const unsigned long long nmk = nL != kNil ? g.lmark[nL] : 0;
        uint32_t dx[kMaxMulti];
        bool any = false;
#pragma unroll
        for (uint32_t j = 0; j < kMaxMulti; ++j) {
            dx[j] = (j < m.k && L != kNil) ? node_dist(__ldcg(&m.c[j].D[src])) : kInf32;
            any |= dx[j] != kInf32;
        }
        const uint32_t mlane = (uint32_t)(mk & 0xFF);
        const uint32_t first_lane = mlane == kInvalidLane ? 32u : mlane;
        const bool go = L != kNil && any;
        const uint32_t start = go ? (uint32_t)(mk >> 32) : kNil;
        uint4 lo, hi;
        group4_load(g, start, lo, hi);
        lists += __popc(__ballot_sync(kFull, go && s4 == 0));
        const uint32_t x = src;
        slabs += walk_lists_g4_from(g, start, true, lo, hi, first_lane, m.c[0].max_hops,
                                    [&](const uint32_t(&y)[4], const uint32_t(&w)[4], const bool(&live)[4]) {
                                        for (uint32_t j = 0; j < m.k; ++j) {
                                            const RoundArgs &a = m.c[j];
                                            relax_edges4(a, x, dx[j], y, w, live, round[j], bqs[j], a.front[0],
                                                         a.ctr + kCnt0, (int *)(a.ctr + kOverflow), edges,
                                                         improved);
                                        }
                                    });
        L = nL;
        nL = nnL;
        src = nsrc;
        mk = nmk;
    }
    for (uint32_t j = 0; j < m.k; ++j)
        frontier_flush(bqs[j], m.c[j].front[0], m.c[j].ctr + kCnt0, m.c[j].cap, (int *)(m.c[j].ctr + kOverflow));
    count_add(g.st, kCtrSeedLists, lists);
    count_add(g.st, kCtrSeedSlabs, slabs);
    count_add(g.st, kCtrSeedEdges, warp_sum(edges));
    count_add(g.st, kCtrSeedImproved, warp_sum(improved));
}

// The decremental relax-into-invalid scan (k_relax_into_invalid_slabs) for
// every state at once (scan_slab_chunks: 32-slab chunks, of which only the
// slabs kept are staged in shared memory by bulk copies): a slab is staged
// when its source has a finite distance in any state that invalidated something, and its live pairs are
// then tested against each such state's invalidation bitmap.
__global__ void __launch_bounds__(kScanWarps * 32) k_relax_into_invalid_multi(MultiArgs m)
{
    __shared__ ScanSmem sm;
    const GView &g = m.c[0].g;
    bool act[kMaxMulti];
    bool any_act = false;
#pragma unroll
    for (uint32_t j = 0; j < kMaxMulti; ++j) {
        act[j] = j < m.k && __ldg(m.c[j].ctr + kInvTotal) != 0;
        any_act |= act[j];
    }
    if (!any_act)
        return;
    const uint32_t lane = lane_id();
    uint32_t slabs = 0, edges = 0, owners = 0, targets = 0;
    const bool ok = scan_slab_chunks(
        g, sm,
        [&](uint32_t own) {
            owners += own != kNil;
            uint4 dx = make_uint4(kInf32, kInf32, kInf32, kInf32);
            if (own != kNil) {
                dx.x = act[0] ? node_dist(__ldcg(&m.c[0].D[own])) : kInf32;
                dx.y = act[1] ? node_dist(__ldcg(&m.c[1].D[own])) : kInf32;
                dx.z = act[2] ? node_dist(__ldcg(&m.c[2].D[own])) : kInf32;
                dx.w = act[3] ? node_dist(__ldcg(&m.c[3].D[own])) : kInf32;
            }
            return dx;
        },
        [](const uint4 &dx) { return dx.x != kInf32 || dx.y != kInf32 || dx.z != kInf32 || dx.w != kInf32; },
        [&](const uint4 *buf, const uint8_t *comp, uint32_t n, uint32_t own_l, const uint4 &dx_l) {
            const bool active = lane < n;
            const uint32_t it = active ? comp[lane] : 0u;
            const uint32_t own = __shfl_sync(kFull, own_l, it);
            const uint32_t dxs[kMaxMulti] = {__shfl_sync(kFull, dx_l.x, it), __shfl_sync(kFull, dx_l.y, it),
                                             __shfl_sync(kFull, dx_l.z, it), __shfl_sync(kFull, dx_l.w, it)};
            slabs += active;
            if (!__any_sync(kFull, active))
                return;
            const uint32_t *mine = reinterpret_cast<const uint32_t *>(buf + (active ? lane : 0) * 8);
            uint32_t key[16];
            uint32_t live = 0;
#pragma unroll
            for (int q = 0; q < 8; ++q) {
                const uint32_t qq = (q + lane) & 7u;
                const uint4 v = reinterpret_cast<const uint4 *>(mine)[qq];
                const bool l0 = active && v.x < kTombKey, l1 = active && qq != 7u && v.z < kTombKey;
                key[2 * q] = v.x;
                key[2 * q + 1] = v.z;
                live |= (l0 ? 1u : 0u) << (2 * q) | (l1 ? 1u : 0u) << (2 * q + 1);
            }
            edges += __popc(live);
            for (uint32_t j = 0; j < m.k; ++j) {
                const RoundArgs &a = m.c[j];
                const uint32_t dx = dxs[j];
                const uint32_t lj = dx != kInf32 ? live : 0u;
                if (!__any_sync(kFull, lj != 0))
                    continue;
                uint32_t word[16];
#pragma unroll
                for (int k = 0; k < 16; ++k)
                    word[k] = ((lj >> k) & 1u) ? __ldg(&a.inv[key[k] >> 5]) : 0u;
                uint32_t hit = 0;
#pragma unroll
                for (int k = 0; k < 16; ++k)
                    hit |= ((word[k] >> (key[k] & 31u)) & 1u) << k;
                hit &= lj;
                targets += __popc(hit);
                while (hit) {
                    const int k = __ffs(hit) - 1;
                    hit &= hit - 1;
                    const uint32_t at = (((uint32_t)(k >> 1) + lane) & 7u) * 4 + 2 * (k & 1);
                    const unsigned long long nd = (unsigned long long)dx + (a.unit ? 1u : mine[at + 1]);
                    if (nd < kInf32)
                        atomicMin(&a.D[mine[at]], (nd << 32) | own);
                }
            }
        });
    if (!ok)
        set_status(g.st, kErrTimeout);
    count_add(g.st, kCtrScanOwners, __reduce_add_sync(kFull, owners));
    count_add(g.st, kCtrScanSlabs, __reduce_add_sync(kFull, slabs));
    count_add(g.st, kCtrScanEdges, __reduce_add_sync(kFull, edges));
    count_add(g.st, kCtrScanTargets, __reduce_add_sync(kFull, targets));
}

// The round loop of every state in one cooperative launch: in round r each
// state with a non-empty frontier is relaxed over the whole grid (one state
// after another), then one grid barrier ends the round for all of them; the
// loop ends when every frontier is empty.  Block 0 clears each state's
// counter for round r + 2 every round, so a state whose frontier emptied
// keeps reading zero.  No solo phase: rounds of a few lists cost a grid
// barrier each.  Then every state's epilogue (dist/parent, round stamp).
// Dynamic shared memory: one staging area per state.
__global__ void __launch_bounds__(kRoundsMaxThreads, 1) k_rounds_multi(MultiArgs m)
{
    extern __shared__ unsigned char multi_smem[];
    auto *bqs = reinterpret_cast<FrontierSmem<kRoundsMaxThreads / 32> *>(multi_smem);
    __shared__ uint32_t s_n[kMaxMulti];
    for (uint32_t j = 0; j < m.k; ++j)
        frontier_init(bqs[j]);
    const uint64_t warp0 = (uint64_t)(threadIdx.x >> 5) * gridDim.x + blockIdx.x; // as in k_rounds
    const uint64_t nwarps = ((uint64_t)gridDim.x * blockDim.x) >> 5;
    const RoundArgs &a0 = m.c[0];
    uint32_t r = 0, bars = 0, passed = 0;
    bool ok = true;
    while (r < a0.max_rounds) {
        if (threadIdx.x == 0)
            for (uint32_t j = 0; j < m.k; ++j)
                s_n[j] = min(ld_volatile(count_of(m.c[j].ctr, r)), m.c[j].cap);
        __syncthreads();
        uint32_t total = 0;
        for (uint32_t j = 0; j < m.k; ++j)
            total += s_n[j];
        if (total == 0)
            break;
        if (blockIdx.x == 0 && threadIdx.x == 0)
            for (uint32_t j = 0; j < m.k; ++j)
                *count_of(m.c[j].ctr, r + 2) = 0;
        for (uint32_t j = 0; j < m.k; ++j) {
            const uint32_t n = s_n[j];
            if (n == 0)
                continue;
            const RoundArgs &a = m.c[j];
            const uint32_t in = r & 1;
            unsigned long long *cnt = count_of(a.ctr, r + 1);
            relax_body(a, a.front[in], n, a.front[in ^ 1], cnt, __ldg(a.ctr + kRid) + 2 + r, warp0, nwarps,
                       kDirectLists, bqs[j]);
            frontier_flush(bqs[j], a.front[in ^ 1], cnt, a.cap, (int *)(a.ctr + kOverflow));
        }
        ++bars;
        if (!grid_barrier(a0.ctr + kBar, passed, a0.barrier_spins)) {
            ok = false;
            break;
        }
        ++r;
    }
    const uint64_t stride = (uint64_t)gridDim.x * blockDim.x;
    for (uint32_t j = 0; j < m.k; ++j) {
        const RoundArgs &a = m.c[j];
        if (a.dist || a.parent)
            for (uint64_t v = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; v < a.g.V; v += stride) {
                const unsigned long long d = __ldcg(&a.D[v]);
                if (a.dist)
                    a.dist[v] = node_dist(d);
                if (a.parent)
                    a.parent[v] = node_parent(d);
            }
    }
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        bool bad = !ok || r >= a0.max_rounds;
        for (uint32_t j = 0; j < m.k; ++j) {
            const RoundArgs &a = m.c[j];
            a.ctr[kRoundsDone] = r;
            a.ctr[kRid] += r + 2;
            if (a.dist || a.parent)
                atomicAdd(&a.g.st->ctr[kCtrUnpacked][0], (unsigned long long)a.g.V);
            bad |= ld_volatile(a.ctr + kOverflow) != 0;
        }
        atomicAdd(&a0.g.st->ctr[kCtrRounds][0], (unsigned long long)r);
        atomicAdd(&a0.g.st->ctr[kCtrGridBarriers][0], (unsigned long long)bars);
        if (bad)
            set_status(a0.g.st, kErrTimeout);
    }
}

// ---------------------------------------------------------------- host side

namespace {

mk_status get_consumer(mk_graph *g, int kind, uint32_t source, cudaStream_t s, Consumer **out)
{
    auto key = std::make_pair(kind, source);
    auto it = g->consumers.find(key);
    if (it != g->consumers.end()) {
        *out = it->second;
        return MK_OK;
    }
    Consumer *c = new Consumer;
    c->kind = kind;
    c->source = source;
    const size_t V = g->v.V, H = g->v.H;
    mk_status st = device_alloc(g, (void **)&c->D, V * 8, s);
    if (st == MK_OK)
        st = device_alloc(g, (void **)&c->front[0], H * 8, s);
    if (st == MK_OK)
        st = device_alloc(g, (void **)&c->front[1], H * 8, s);
    // frontier slots hold <kNil, ...> until written, so a slot read before
    // it is written names no list
    if (st == MK_OK && (cudaMemsetAsync(c->front[0], 0xFF, H * 8, s) != cudaSuccess ||
                        cudaMemsetAsync(c->front[1], 0xFF, H * 8, s) != cudaSuccess))
        st = MK_ERR_CUDA;
    if (st == MK_OK)
        st = device_alloc(g, (void **)&c->stamp, V * 4, s);
    if (st == MK_OK)
        st = device_alloc(g, (void **)&c->inv, (V + 31) / 32 * 4, s);
    if (st == MK_OK)
        st = device_alloc(g, (void **)&c->counters, kConsumerWords * 4, s);
    if (st == MK_OK && (cudaMemsetAsync(c->stamp, 0, V * 4, s) != cudaSuccess || cudaMemsetAsync(c->counters, 0, kConsumerWords * 4, s) != cudaSuccess))
        st = MK_ERR_CUDA;
    if (st != MK_OK) {
        device_free(g, c->D, V * 8, s);
        device_free(g, c->front[0], H * 8, s);
        device_free(g, c->front[1], H * 8, s);
        device_free(g, c->stamp, V * 4, s);
        device_free(g, c->inv, (V + 31) / 32 * 4, s);
        device_free(g, c->counters, kConsumerWords * 4, s);
        delete c;
        return st;
    }
    g->consumers[key] = c;
    *out = c;
    return MK_OK;
}

} // namespace

namespace mk {

// The persistent round kernel runs one block per SM; the tuned value
// (rounds_blocks_per_sm) is the block size in units of 256 threads, at most
// what fits an SM (the occupancy of 256-thread blocks).  One block per SM
// keeps the grid barrier to one arrival per SM and gives the solo rounds
// the whole SM.
int rounds_max_blocks_per_sm()
{
    static int per = 0;
    if (!per) {
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, k_rounds<false>, 256, 0);
        per = std::min(std::max(per, 1), (int)(kRoundsMaxThreads / 256));
    }
    return per;
}

int rounds_grid(int) { return num_sms(); }

int rounds_block(int units)
{
    const int max_units = rounds_max_blocks_per_sm();
    return 256 * (units > 0 ? std::min(units, max_units) : max_units);
}

} // namespace mk

namespace {

// Runs every round of one phase and the call's epilogue (round stamp,
// overflow check, a.dist / a.parent written from D).  Input: front[0], size
// in ctr[kCnt0], the rotating pairs zero.
mk_status run_phase(mk_graph *g, RoundArgs a, const char *name, cudaStream_t s)
{
    const int grid = rounds_grid(g->tune.rounds_blocks_per_sm);
    const int block = rounds_block(g->tune.rounds_blocks_per_sm);
    void *args[] = {&a};
    if (!g->dbg_host_rounds) {
        const mk_status st = timed(g, name, s, 1, [&]() {
            const void *k = a.delta ? (const void *)k_rounds<true> : (const void *)k_rounds<false>;
            return cudaLaunchCooperativeKernel(k, dim3(grid), dim3(block), args, 0, s);
        });
        if (st == MK_OK)
            return MK_OK;
        cudaGetLastError();
    }
    // fallback: one launch per round, the host reads each size
    for (uint32_t r = 0;; ++r) {
        if (r > a.max_rounds)
            return MK_ERR_TIMEOUT;
        MK_CUDA(cudaMemcpyAsync(g->h_pinned, count_of(a.ctr, r), 4, cudaMemcpyDeviceToHost, s));
        MK_CUDA(cudaStreamSynchronize(s));
        const uint32_t n = std::min(g->h_pinned[0], a.cap);
        if (n == 0) {
            return timed(g, "sssp_finish", s, 2, [&]() {
                k_sssp_finish<<<1, 1, 0, s>>>(a.ctr, g->d_state, r);
                if (a.dist || a.parent)
                    k_unpack<<<grid_for(a.g.V, 256), 256, 0, s>>>(a.D, a.g.V, a.dist, a.parent);
                return cudaSuccess;
            });
        }
        MK_TRY(timed(g, name, s, 1, [&]() {
            k_round_once<<<grid_for((uint64_t)n, 256), 256, 0, s>>>(a, r, n);
            return cudaSuccess;
        }));
    }
}

mk_status run_sssp(mk_graph *g, int kind, uint32_t source, uint32_t *d_dist, uint32_t *d_parent, cudaStream_t s)
{
    if (!g || source >= g->v.V)
        return MK_ERR_INVALID_ARG;
    Consumer *c = nullptr;
    MK_TRY(get_consumer(g, kind, source, s, &c));
    const uint32_t V = g->v.V, H = g->v.H;
    RoundArgs a{};
    a.g = g->v;
    a.D = c->D;
    a.front[0] = c->front[0];
    a.front[1] = c->front[1];
    a.ctr = c->counters;
    a.stamp = c->stamp;
    a.inv = c->inv;
    a.cap = H;
    a.max_hops = g->v.P + 2;
    a.max_rounds = V + 2;
    a.barrier_spins = g->dbg_barrier_spins != ~0ull ? (uint32_t)g->dbg_barrier_spins : kBarrierSpins;
    a.source = source;
    a.unit = kind == kBfs ? 1 : 0;
    a.dist = d_dist;
    a.parent = d_parent;
    const bool incremental = c->epoch == g->epoch;
    // Near-Far ordering for SSSP when a bucket width is set for this kind of
    // call (the host-driven fallback runs plain rounds)
    a.delta = kind == kSssp && !g->dbg_host_rounds ? (incremental ? g->sssp_delta_incr : g->sssp_delta_static) : 0;
    if (a.delta && !c->fstamp) {
        mk_status st = device_alloc(g, (void **)&c->far[0], (size_t)V * 4, s);
        if (st == MK_OK)
            st = device_alloc(g, (void **)&c->far[1], (size_t)V * 4, s);
        if (st == MK_OK)
            st = device_alloc(g, (void **)&c->fstamp, (size_t)V * 4, s);
        if (st == MK_OK && cudaMemsetAsync(c->fstamp, 0, (size_t)V * 4, s) != cudaSuccess)
            st = MK_ERR_CUDA;
        if (st != MK_OK) {
            device_free(g, c->far[0], (size_t)V * 4, s);
            device_free(g, c->far[1], (size_t)V * 4, s);
            device_free(g, c->fstamp, (size_t)V * 4, s);
            c->far[0] = c->far[1] = c->fstamp = nullptr;
            return st;
        }
    }
    a.far[0] = c->far[0];
    a.far[1] = c->far[1];
    a.fstamp = c->fstamp;
    MK_CUDA(cudaMemsetAsync(c->counters, 0, kClearWords * 4, s));
    if (a.delta) // the piles' minima and first rounds, and the first frontier's minimum, at INF
        MK_CUDA(cudaMemsetAsync(c->counters + kFarMin0, 0xFF, kOrderWords * 4, s));
    if (!incremental) {
        MK_TRY(timed(g, "sssp_init", s, 1, [&]() {
            k_sssp_init<<<grid_for(V, 256), 256, 0, s>>>(c->D, V, source, c->front[0], c->counters + kCnt0,
                                                         g->v.vinfo);
            return cudaSuccess;
        }));
    } else {
        if (g->epoch_has_deletes) {
            // decremental prologue: invalidate, spread down the tree, then
            // relax the edges from valid into invalidated vertices
            MK_CUDA(cudaMemsetAsync(c->inv, 0, (size_t)(V + 31) / 32 * 4, s));
            MK_TRY(timed(g, "sssp_invalidate", s, 1, [&]() {
                k_invalidate<<<grid_for(std::max<uint64_t>(g->dlog_bound, 1), 256), 256, 0, s>>>(g->d_dlog,
                                                                                                 g->dlog_bound, a);
                return cudaSuccess;
            }));
            MK_TRY(timed(g, "sssp_invalidate_walk", s, 1, [&]() {
                k_inv_walk<<<grid_for(V, 256), 256, 0, s>>>(a);
                return cudaSuccess;
            }));
            MK_TRY(timed(g, "sssp_relax_into_invalid", s, 1, [&]() {
                const size_t bytes = ((size_t)V + 31) / 32 * 4;
                constexpr size_t kMost = 200u << 10;
                if (bytes > kMost) {
                    k_relax_into_invalid_slabs<2><<<num_sms(), kInvThreads, 0, s>>>(a);
                    return cudaSuccess;
                }
                auto k = k_relax_into_invalid_slabs<1>;
                // (not `bytes`: another thread may be about to launch it for a larger graph)
                const cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kMost);
                if (e != cudaSuccess)
                    return e;
                k<<<num_sms(), kInvThreads, bytes, s>>>(a);
                return cudaSuccess;
            }));
            MK_TRY(timed(g, "sssp_enqueue_invalid", s, 1, [&]() {
                k_enqueue_invalid<<<grid_for(((uint64_t)V + 31) / 32 * 32, 256), 256, 0, s>>>(a);
                return cudaSuccess;
            }));
        }
        // incremental prologue: edges inserted since the last commit, from
        // the inserted-edge log when the epoch holds no deletes (every
        // logged edge still live), else by walking the updated lists from
        // their UpdateIterator markers
        if (g->ulog_bound && !g->epoch_has_deletes && g->ilog_ok && g->d_ilog) {
            MK_TRY(timed(g, "sssp_relax_updated", s, 1, [&]() {
                const uint64_t threads = (g->ilog_bound + 3) / 4;
                k_relax_inserted<<<std::min<uint32_t>(grid_for(threads, 256), num_sms() * 8), 256, 0, s>>>(
                    a, g->d_ilog, g->ilog_bound);
                return cudaSuccess;
            }));
        } else if (g->ulog_bound) {
            MK_TRY(timed(g, "sssp_relax_updated", s, 1, [&]() {
                // one 4-lane group per logged list
                const uint64_t threads = g->ulog_bound * 4;
                k_relax_updated<<<std::min<uint32_t>(grid_for(threads, 256), num_sms() * 10), 256, 0, s>>>(a);
                return cudaSuccess;
            }));
        }
    }
    // common epilogue: rounds until no distance improves, then the outputs
    MK_TRY(run_phase(g, a, "sssp_rounds", s));
    c->epoch = g->epoch;
    c->seq = g->change_seq;
    return MK_OK;
}


// Several BFS/SSSP states of one graph in one call (see k_rounds_multi).
mk_status run_multi(mk_graph *g, const mk_algo_req *reqs, uint32_t n, cudaStream_t s)
{
    MultiArgs m{};
    m.k = n;
    Consumer *cs[kMaxMulti] = {};
    bool incr[kMaxMulti] = {};
    const uint32_t V = g->v.V, H = g->v.H;
    for (uint32_t j = 0; j < n; ++j) {
        const int kind = reqs[j].kind == MK_REQ_BFS ? kBfs : kSssp;
        MK_TRY(get_consumer(g, kind, reqs[j].source, s, &cs[j]));
        Consumer *c = cs[j];
        RoundArgs &a = m.c[j];
        a.g = g->v;
        a.D = c->D;
        a.front[0] = c->front[0];
        a.front[1] = c->front[1];
        a.ctr = c->counters;
        a.stamp = c->stamp;
        a.inv = c->inv;
        a.cap = H;
        a.max_hops = g->v.P + 2;
        a.max_rounds = V + 2;
        a.barrier_spins = g->dbg_barrier_spins != ~0ull ? (uint32_t)g->dbg_barrier_spins : kBarrierSpins;
        a.source = reqs[j].source;
        a.unit = kind == kBfs ? 1 : 0;
        a.dist = reqs[j].d_dist;
        a.parent = reqs[j].d_parent;
        incr[j] = c->epoch == g->epoch;
        MK_CUDA(cudaMemsetAsync(c->counters, 0, kClearWords * 4, s));
    }
    // the states that recompute statically start from their sources
    for (uint32_t j = 0; j < n; ++j)
        if (!incr[j])
            MK_TRY(timed(g, "sssp_init", s, 1, [&]() {
                k_sssp_init<<<grid_for(V, 256), 256, 0, s>>>(cs[j]->D, V, m.c[j].source, cs[j]->front[0],
                                                             cs[j]->counters + kCnt0, g->v.vinfo);
                return cudaSuccess;
            }));
    // decremental prologue: invalidation per state, one scan for all
    MultiArgs dec{};
    MultiArgs inc{};
    for (uint32_t j = 0; j < n; ++j)
        if (incr[j]) {
            if (g->epoch_has_deletes)
                dec.c[dec.k++] = m.c[j];
            if (g->ulog_bound)
                inc.c[inc.k++] = m.c[j];
        }
    for (uint32_t j = 0; j < dec.k; ++j) {
        const RoundArgs &a = dec.c[j];
        MK_CUDA(cudaMemsetAsync(a.inv, 0, (size_t)(V + 31) / 32 * 4, s));
        MK_TRY(timed(g, "sssp_invalidate", s, 1, [&]() {
            k_invalidate<<<grid_for(std::max<uint64_t>(g->dlog_bound, 1), 256), 256, 0, s>>>(g->d_dlog, g->dlog_bound,
                                                                                             a);
            return cudaSuccess;
        }));
        MK_TRY(timed(g, "sssp_invalidate_walk", s, 1, [&]() {
            k_inv_walk<<<grid_for(V, 256), 256, 0, s>>>(a);
            return cudaSuccess;
        }));
    }
    if (dec.k) {
        MK_TRY(timed(g, "sssp_relax_into_invalid", s, 1, [&]() {
            static const uint32_t grid = resident_grid(k_relax_into_invalid_multi, kScanWarps * 32);
            k_relax_into_invalid_multi<<<grid, kScanWarps * 32, 0, s>>>(dec);
            return cudaSuccess;
        }));
        for (uint32_t j = 0; j < dec.k; ++j)
            MK_TRY(timed(g, "sssp_enqueue_invalid", s, 1, [&]() {
                k_enqueue_invalid<<<grid_for(((uint64_t)V + 31) / 32 * 32, 256), 256, 0, s>>>(dec.c[j]);
                return cudaSuccess;
            }));
    }
    // incremental prologue: one walk over the updated lists for all states
    if (inc.k) {
        const size_t smem = inc.k * sizeof(FrontierSmem<8>);
        // (a function attribute of the current device: set on every call)
        MK_CUDA(cudaFuncSetAttribute(k_relax_updated_multi, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                     (int)(kMaxMulti * sizeof(FrontierSmem<8>))));
        MK_TRY(timed(g, "sssp_relax_updated", s, 1, [&]() {
            const uint64_t threads = g->ulog_bound * 4;
            k_relax_updated_multi<<<std::min<uint32_t>(grid_for(threads, 256), num_sms() * 10), 256, smem, s>>>(inc);
            return cudaSuccess;
        }));
    }
    // rounds of every state together
    const int grid = rounds_grid(g->tune.rounds_blocks_per_sm);
    const int block = rounds_block(g->tune.rounds_blocks_per_sm);
    const size_t smem = n * sizeof(FrontierSmem<kRoundsMaxThreads / 32>);
    MK_CUDA(cudaFuncSetAttribute(k_rounds_multi, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 (int)(kMaxMulti * sizeof(FrontierSmem<kRoundsMaxThreads / 32>))));
    void *args[] = {&m};
    mk_status st = MK_ERR_CUDA;
    if (!g->dbg_host_rounds)
        st = timed(g, "sssp_rounds", s, 1, [&]() {
            return cudaLaunchCooperativeKernel((const void *)k_rounds_multi, dim3(grid), dim3(block), args, smem, s);
        });
    if (st != MK_OK) {
        cudaGetLastError();
        // one state at a time (the host-driven loop when the cooperative
        // launch is refused)
        for (uint32_t j = 0; j < n; ++j)
            MK_TRY(run_phase(g, m.c[j], "sssp_rounds", s));
    }
    for (uint32_t j = 0; j < n; ++j) {
        cs[j]->epoch = g->epoch;
        cs[j]->seq = g->change_seq;
    }
    return MK_OK;
}
} // namespace

namespace mk {

// Duration of one static BFS from `source` (CUDA events on s), for the
// autotuner; leaves a valid BFS state for that source.
mk_status time_static_bfs(mk_graph *g, uint32_t source, cudaStream_t s, float *ms)
{
    Consumer *c = nullptr;
    MK_TRY(get_consumer(g, kBfs, source, s, &c));
    c->epoch = ~0ull;
    cudaEvent_t a, b;
    MK_CUDA(cudaEventCreate(&a));
    MK_CUDA(cudaEventCreate(&b));
    cudaEventRecord(a, s);
    mk_status st = run_sssp(g, kBfs, source, nullptr, nullptr, s);
    cudaEventRecord(b, s);
    cudaEventSynchronize(b);
    cudaEventElapsedTime(ms, a, b);
    cudaEventDestroy(a);
    cudaEventDestroy(b);
    return st;
}

} // namespace mk

extern "C" {

mk_status mk_incr_sssp(mk_graph *g, uint32_t source, uint32_t *d_dist, uint32_t *d_parent, void *stream)
{
    return run_sssp(g, kSssp, source, d_dist, d_parent, (cudaStream_t)stream);
}

mk_status mk_incr_bfs(mk_graph *g, uint32_t source, uint32_t *d_dist, uint32_t *d_parent, void *stream)
{
    return run_sssp(g, kBfs, source, d_dist, d_parent, (cudaStream_t)stream);
}

mk_status mk_incr_multi(mk_graph *g, const mk_algo_req *h_reqs, uint32_t n, void *stream)
{
    if (!g || !h_reqs || n == 0 || n > kMaxMulti)
        return MK_ERR_INVALID_ARG;
    for (uint32_t j = 0; j < n; ++j) {
        if ((h_reqs[j].kind != MK_REQ_SSSP && h_reqs[j].kind != MK_REQ_BFS) || h_reqs[j].source >= g->v.V)
            return MK_ERR_INVALID_ARG;
        for (uint32_t i = 0; i < j; ++i)
            if (h_reqs[i].kind == h_reqs[j].kind && h_reqs[i].source == h_reqs[j].source)
                return MK_ERR_INVALID_ARG; // one state cannot be advanced twice at once
    }
    cudaStream_t s = (cudaStream_t)stream;
    if (n == 1)
        return run_sssp(g, h_reqs[0].kind == MK_REQ_BFS ? kBfs : kSssp, h_reqs[0].source, h_reqs[0].d_dist,
                        h_reqs[0].d_parent, s);
    return run_multi(g, h_reqs, n, s);
}

} // extern "C"
