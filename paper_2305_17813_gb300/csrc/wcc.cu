// Static and incremental weakly connected components (paper, Sec.
// "Incremental WCC" and Sec. "Auxiliary Data Structures", Union-Find).
//
// Union-Async: to unite sets, find their roots and hook the larger root under
// the smaller with one CAS, retrying with fresh roots when the CAS loses.
// Parents therefore never exceed their child's id, the root of every tree is
// its smallest vertex, and after full path compression each label is the
// smallest vertex id of its component.  Finds use path halving.  A warp unites
// a whole slab at once: the source and the slab's live destinations are
// hooked under the smallest of their roots (one parallel round of finds and
// CASes per slab instead of one union per edge on the same source root), and
// a warp walks eight lists at a time (incremental pass) or eight slabs (static
// pass; four of the set layout).
//
// Static pass: every live edge of every list, most of them settled by a
// sampled forest (below; the set layout's components run here too).
// Incremental pass (insert-only
// epochs): only the entries written since the last commit, read with the
// UpdateIterator from each updated list's marker (the paper's
// ApplyUnionUpdate, which skips lanes before the first updated lane).
#include "mk_host.h"
#include "uf.cuh"
#include "walk.cuh"

#include <algorithm>

using namespace mk;

namespace {

__device__ __forceinline__ uint32_t uf_find(uint32_t *p, uint32_t x)
{
    for (;;) {
        const uint32_t px = __ldcg(&p[x]);
        if (px == x || px == 0) // vertex 0 is always a root
            return px;
        const uint32_t ppx = __ldcg(&p[px]);
        if (ppx == px)
            return px; // px is the root: no third load
        p[x] = ppx;    // path halving: ppx is an ancestor of x
        x = ppx;
    }
}


} // namespace

__global__ void k_uf_init(uint32_t *p, uint32_t V)
{
    const uint32_t v = blockIdx.x * blockDim.x + threadIdx.x;
    if (v < V)
        p[v] = v;
}

// Incremental pass: unites the source of every list in the updated-list log
// with the destinations inserted since the last commit, read with the
// UpdateIterator from the list's marker (the marker slab's lanes before the
// marker lane are skipped; a full marker slab is skipped entirely).  Every
// 4-lane group of every warp takes one list at a time (group index + k *
// groups in the grid; eight lists per warp) and walks it with two 16-byte
// loads per lane (pairs 4*s4 .. 4*s4+3); the unused slot of lane 3 (slab
// lane 30) carries the list's source, so each slab's source and
// destinations are united in one group_union.  The next list's log entry,
// source and marker are loaded a step ahead.
__global__ void __launch_bounds__(256, 5) k_uf_hook(GView g, uint32_t *p, uint32_t max_hops, int *failed)
{
    const uint32_t lane = lane_id(), gi = lane >> 2, s4 = lane & 3u, gbase = lane & ~3u;
    const uint32_t n = min(__ldg(&g.st->ulog_count), g.H);
    const uint64_t warp0 = (blockIdx.x * (uint64_t)blockDim.x + threadIdx.x) >> 5;
    const uint64_t gs = (((uint64_t)gridDim.x * blockDim.x) >> 5) * 8;
    unsigned long long slabs = 0, edges = 0;
    uint64_t i = warp0 * 8 + gi;
    uint32_t L = i < n ? g.ulog[i] : kNil;
    uint32_t nL = i + gs < n ? g.ulog[i + gs] : kNil;
    uint32_t src = L != kNil ? g.list_src[L] : 0;
    unsigned long long mk = L != kNil ? g.lmark[L] : 0;
    for (uint64_t base = warp0 * 8; base < n; base += gs, i += gs) {
        const uint32_t nnL = i + 2 * gs < n ? g.ulog[i + 2 * gs] : kNil;
        const uint32_t nsrc = nL != kNil ? g.list_src[nL] : 0;
        const unsigned long long nmk = nL != kNil ? g.lmark[nL] : 0;
        const uint32_t mlane = (uint32_t)(mk & 0xFF);
        uint32_t first_lane = mlane == kInvalidLane ? 32u : mlane;
        uint32_t slab = L != kNil ? (uint32_t)(mk >> 32) : kNil;
        bool active = slab != kNil;
        for (uint32_t hop = 0; __any_sync(kFull, active); ++hop) {
            uint4 lo = make_uint4(kEmptyKey, kFull, kFull, kFull), hi = lo;
            if (active) {
                const uint4 *q = reinterpret_cast<const uint4 *>(slab_ptr(g, slab) + s4 * 8);
                lo = __ldcg(q);
                hi = __ldcg(q + 1);
            }
            slabs += __popc(__ballot_sync(kFull, active && s4 == 0));
            const bool last = s4 == 3u;
            const uint32_t w0 = 8 * s4;
            const uint32_t e[4] = {lo.x, lo.z, hi.x, last ? src : hi.z};
            const bool act[4] = {active && lo.x < kTombKey && w0 >= first_lane,
                                 active && lo.z < kTombKey && w0 + 2 >= first_lane,
                                 active && hi.x < kTombKey && w0 + 4 >= first_lane,
                                 last ? active : (active && hi.z < kTombKey && w0 + 6 >= first_lane)};
            edges += __popc(__ballot_sync(kFull, act[0])) + __popc(__ballot_sync(kFull, act[1])) +
                     __popc(__ballot_sync(kFull, act[2])) + __popc(__ballot_sync(kFull, act[3] && !last));
            if (!group_union<4, 4>(p, e, act, 1u << 20) && lane == 0)
                *failed = 1;
            const uint32_t nxt = __shfl_sync(kFull, hi.w, gbase + 3);
            if (active) {
                if (nxt == kNil || hop + 1 >= max_hops)
                    active = false;
                else
                    slab = nxt;
            }
            first_lane = 0;
        }
        L = nL;
        nL = nnL;
        src = nsrc;
        mk = nmk;
    }
    count_add(g.st, kCtrWccUpdSlabs, slabs);
    count_add(g.st, kCtrWccUpdEdges, edges);
}

// Incremental pass from the inserted-edge log (insert-only epochs, so every
// logged edge is live): each lane unites the two ends of one logged edge
// (a one-lane group_union: both roots found in lockstep, the larger hooked
// under the smaller).
__global__ void __launch_bounds__(256) k_uf_hook_log(DevState *st, const uint4 *__restrict__ ilog, uint64_t n,
                                                     uint32_t *p, int *failed)
{
    const uint64_t stride = (uint64_t)gridDim.x * blockDim.x;
    unsigned long long entries = 0;
    for (uint64_t wb = (blockIdx.x * (uint64_t)blockDim.x + threadIdx.x) & ~31ull; wb < n; wb += stride) {
        const uint64_t i = wb + lane_id();
        const uint4 e = i < n ? __ldcs(&ilog[i]) : make_uint4(kNil, 0, 0, 0); // kNil: nothing was stored
        const uint32_t x[2] = {e.x, e.y};
        const bool act[2] = {e.x != kNil, e.x != kNil};
        entries += __popc(__ballot_sync(kFull, act[0]));
        if (!group_union<1, 2>(p, x, act, 1u << 20) && lane_id() == 0)
            *failed = 1;
    }
    count_add(st, kCtrWccLog, entries);
    count_add(st, kCtrWccUpdEdges, entries);
}

// ------------------------------------------------------------- static pass
//
// Most edges of most graphs lie inside one component, and finding that out
// edge by edge is what the pass cost: two finds each, ending in the same few
// roots, and hooks that lose to one another there (168-194 us on an R-MAT
// graph of scale 18 whose slabs are read in 12).  So the pass first builds a
// forest from a sample -- the first four or so keys of every vertex's first
// list (sample_of): every vertex points to its smallest sampled neighbour
// below it, the trees are compressed, the roots that sampled edges connect
// are hooked with plain atomic minima, and the trees are compressed again.
// The tree that holds most of 1,024 sampled vertices is the giant one; a
// bitmap names its vertices.  The scan over all slabs then tests both ends of an edge in the bitmap, which it keeps in
// shared memory where it fits, and only slabs with an edge that is not inside
// the giant tree unite anything.  Kernel boundaries in between also drop the
// parents that the SMs' L1 caches still hold from before the hooks.
// (The order of things -- sampled neighbours, link, compress, most frequent tree,
// then what lies outside it -- is Afforest's: Sutton, Ben-Nun and Barak,
// "Optimizing Parallel Graph Connectivity Computation via Subgraph Sampling",
// IPDPS 2018.)
// Sampled hooks may lose a link (a minimum replaces a root's earlier one):
// the forest stays one of connected vertices with parents below their
// children, and the scan looks at every edge again.

namespace {

// One slab is read by eight lanes, 16 bytes each, so that a load covers whole
// sectors: a lane has two keys of the map layout, four of the set's.  The last
// lane's last place is no key (the map's unused lane, the set's next index).
constexpr uint32_t kLanes = 8;

template <bool kSet>
__device__ __forceinline__ void keys_of(const uint4 &q, uint32_t (&e)[kSet ? 4 : 2])
{
    if constexpr (kSet) {
        e[0] = q.x, e[1] = q.y, e[2] = q.z, e[3] = q.w;
    } else {
        e[0] = q.x, e[1] = q.z;
    }
}

// The sampled neighbours of v: f(d) for 32 bytes of its first list at a time
// (d: their keys, kNil where there is none) until four keys were found or the
// list ends.  A new list has them in its first 32 bytes; one that has seen
// deletions starts with tombstones, and a sample of those alone would leave
// the vertex out of its tree and all its edges to the scan (20 batches of
// 2^20 inserts and deletes on R-MAT scale 20: 343 us for the scan instead of
// 110).
template <bool kSet, typename F>
__device__ __forceinline__ void sample_of(const GView &g, uint32_t v, F &&f)
{
    constexpr uint32_t kParts = 32, kEnough = 4; // 8 slabs at most
    uint32_t slab = __ldg(&g.vinfo[v]).x, found = 0;
    for (uint32_t part = 0; part < kParts && found < kEnough; ++part) {
        const uint32_t in = part & 3u;
        const uint4 *p = reinterpret_cast<const uint4 *>(slab_ptr(g, slab)) + 2 * in;
        const uint4 a = __ldcg(p), b = __ldcg(p + 1);
        uint32_t d[8] = {a.x, kSet ? a.y : kNil, a.z, kSet ? a.w : kNil,
                         b.x, kSet ? b.y : kNil, b.z, kSet && in != 3u ? b.w : kNil};
        bool end = false; // keys fill in order: a free one ends the list
#pragma unroll
        for (int k = 0; k < 8; ++k) {
            end = end || d[k] == kEmptyKey;
            d[k] = d[k] < kTombKey ? d[k] : kNil;
            found += d[k] != kNil;
        }
        f(d);
        if (in == 3u)
            slab = b.w;
        if (end || slab == kNil)
            break;
    }
}

} // namespace

template <bool kSet>
__global__ void __launch_bounds__(256) k_cc_sample(GView g, uint32_t *p)
{
    const uint32_t v = blockIdx.x * blockDim.x + threadIdx.x;
    if (v >= g.V)
        return;
    uint32_t m = v;
    sample_of<kSet>(g, v, [&](const uint32_t(&d)[8]) {
#pragma unroll
        for (int k = 0; k < 8; ++k)
            m = min(m, d[k]);
    });
    p[v] = m;
}

// Every kLinkStep-th vertex: enough to hook nearly every root (what is left
// is united in the scan), and few enough at a time that the hooks of the
// larger trees' roots do not queue up on a few words.
constexpr uint32_t kLinkStep = 8;

template <bool kSet>
__global__ void __launch_bounds__(256) k_cc_link(GView g, uint32_t *p)
{
    const uint64_t at = (blockIdx.x * (uint64_t)blockDim.x + threadIdx.x) * kLinkStep;
    if (at >= g.V)
        return;
    const uint32_t v = (uint32_t)at;
    const uint32_t rv = __ldcg(&p[v]);
    sample_of<kSet>(g, v, [&](const uint32_t(&d)[8]) {
        uint32_t r[8];
#pragma unroll
        for (int k = 0; k < 8; ++k)
            r[k] = d[k] != kNil ? __ldcg(&p[d[k]]) : rv;
#pragma unroll
        for (int k = 0; k < 8; ++k) {
            const uint32_t hi = max(r[k], rv), lo = min(r[k], rv);
            if (hi != lo && __ldcg(&p[hi]) > lo)
                atomicMin(&p[hi], lo);
        }
    });
}

// p[v] = v's root for every vertex, and into label where that is given.  Ends
// a pass when `failed` is given: a hook that gave up sets the status.
__global__ void __launch_bounds__(256) k_uf_compress(uint32_t *p, uint32_t V, uint32_t *label, const int *failed,
                                                     DevState *st)
{
    const uint32_t v = blockIdx.x * blockDim.x + threadIdx.x;
    if (failed && v == 0 && *failed)
        set_status(st, kErrTimeout);
    if (v >= V)
        return;
    const uint32_t r = uf_find(p, v);
    p[v] = r;
    if (label)
        label[v] = r;
}

// *giant = the root that most of 1,024 vertices spread over the range have.
__global__ void __launch_bounds__(1024) k_cc_giant(const uint32_t *p, uint32_t V, uint32_t *giant)
{
    __shared__ uint32_t key[2048], cnt[2048], best;
    const uint32_t t = threadIdx.x;
    for (uint32_t i = t; i < 2048; i += 1024) {
        key[i] = kNil;
        cnt[i] = 0;
    }
    if (t == 0)
        best = 0;
    __syncthreads();
    const uint32_t r = __ldcg(&p[(uint32_t)((uint64_t)V * t >> 10)]);
    uint32_t h = hash32(r) & 2047u;
    for (;;) { // at most half full
        const uint32_t own = atomicCAS(&key[h], kNil, r);
        if (own == kNil || own == r)
            break;
        h = (h + 1) & 2047u;
    }
    const uint32_t mine = atomicAdd(&cnt[h], 1u) + 1; // the last of a root counts them all
    atomicMax(&best, mine);
    __syncthreads();
    if (mine == best)
        *giant = r; // of equals, any
}

__global__ void __launch_bounds__(256) k_cc_bits(const uint32_t *p, uint32_t V, const uint32_t *giant, uint32_t *bits)
{
    const uint32_t v = blockIdx.x * blockDim.x + threadIdx.x;
    const uint32_t m = __ballot_sync(kFull, v < V && p[v] == __ldg(giant));
    if (lane_id() == 0 && v < V)
        bits[v >> 5] = m;
}

namespace {

// Edges waiting to be united, a buffer a warp.
constexpr uint32_t kPairBuf = 192; // 63 of the steps before and 128 of this one

// Unites the warp's first min(n, 64) pairs of buf, two a lane, their finds in
// lockstep; a hook that loses is done again one pair at a time.
__device__ __forceinline__ bool unite_pairs(uint32_t *p, const uint2 *buf, uint32_t n)
{
    const uint32_t lane = lane_id();
    uint32_t x[4];
    bool lost[2];
#pragma unroll
    for (uint32_t i = 0; i < 2; ++i) {
        const uint32_t at = lane + 32 * i;
        const uint2 e = at < n ? buf[at] : make_uint2(kNil, kNil);
        x[2 * i] = e.x;
        x[2 * i + 1] = e.y;
    }
    uf_find_n<4, true>(p, x);
#pragma unroll
    for (uint32_t i = 0; i < 2; ++i) {
        const uint32_t hi = max(x[2 * i], x[2 * i + 1]), lo = min(x[2 * i], x[2 * i + 1]);
        lost[i] = hi != lo && atomicCAS(&p[hi], hi, lo) != hi;
    }
    bool ok = true;
#pragma unroll
    for (uint32_t i = 0; i < 2; ++i)
        if (__any_sync(kFull, lost[i])) {
            const uint32_t e[2] = {x[2 * i], x[2 * i + 1]};
            const bool act[2] = {lost[i], lost[i]};
            ok = group_union<1, 2>(p, e, act, 1u << 20) && ok;
        }
    __syncwarp();
    return ok;
}

} // namespace

// The scan: a warp takes 32 consecutive slabs at a time, one a group of
// kLanes lanes: their owners in one load (read a chunk ahead; kNil for an
// unused pool slab), then all of their parts at once.  kBits: 0 unites every
// slab, 1 tests the bitmap in shared memory, 2 in global memory; an edge that
// is not inside the giant tree then waits in a buffer until 64 are there, so
// that the scan does not stop for the round trips of every few.  Bound by
// instructions (R-MAT scale 20: 4.3 % of the edges are united; 91 us for
// 300 MB of slabs).
constexpr uint32_t kScanThreads = 1024;

template <bool kSet, int kBits>
__global__ void __launch_bounds__(kScanThreads, 1) k_cc_scan(GView g, uint32_t *p, const uint32_t *__restrict__ bits,
                                                             const uint32_t *giant, int *failed)
{
    constexpr uint32_t kGroups = 32 / kLanes, kSteps = 32 / kGroups;
    constexpr int kKeys = kSet ? 4 : 2;
    extern __shared__ uint32_t s_bits[];
    __shared__ uint2 pairs[kBits ? kScanThreads / 32 : 1][kBits ? kPairBuf : 1];
    const uint32_t lane = lane_id(), gr = lane / kLanes, sub = lane % kLanes, w = threadIdx.x >> 5;
    const bool last = sub == kLanes - 1;
    const uint32_t root = kBits ? __ldg(giant) : 0u;
    if (kBits == 1) {
        for (uint32_t i = threadIdx.x; i < (g.V + 31) / 32; i += kScanThreads)
            s_bits[i] = __ldg(&bits[i]);
        __syncthreads();
    }
    auto inside = [&](uint32_t v) -> uint32_t {
        return ((kBits == 1 ? s_bits[v >> 5] : __ldg(&bits[v >> 5])) >> (v & 31u)) & 1u;
    };
    const uint64_t total = (uint64_t)g.H + g.P;
    const uint64_t stride = (((uint64_t)gridDim.x * kScanThreads) >> 5) * 32;
    uint32_t slabs = 0, edges = 0; // of this warp, of this lane
    uint32_t held = 0, united = 0; // pairs in the warp's buffer, and taken out of it
    bool ok = true;
    uint64_t c = ((blockIdx.x * (uint64_t)kScanThreads + threadIdx.x) >> 5) * 32;
    uint32_t own_next = c + lane < total ? __ldcg(&g.owner[c + lane]) : kNil;
    for (; c < total; c += stride) {
        const uint32_t own_l = own_next;
        own_next = c + stride + lane < total ? __ldcg(&g.owner[c + stride + lane]) : kNil;
        const uint32_t live = __ballot_sync(kFull, own_l != kNil);
        if (!live)
            continue;
        uint4 part[kSteps];
        const uint4 *at = reinterpret_cast<const uint4 *>(slab_ptr(g, (uint32_t)c + gr)) + sub;
#pragma unroll
        for (uint32_t j = 0; j < kSteps; ++j)
            part[j] = (live >> (j * kGroups + gr)) & 1u ? __ldcg(at + j * kGroups * 8)
                                                        : make_uint4(kEmptyKey, kEmptyKey, kEmptyKey, kEmptyKey);
        const uint32_t in = kBits ? __ballot_sync(kFull, own_l != kNil && inside(own_l)) : 0u;
        slabs += __popc(live);
#pragma unroll
        for (uint32_t j = 0; j < kSteps; ++j) {
            const uint32_t it = j * kGroups + gr;
            uint32_t e[kKeys], keys = 0, out = 0; // bit k: e[k] is a key; and it is outside the giant tree
            keys_of<kSet>(part[j], e);
#pragma unroll
            for (int k = 0; k < kKeys; ++k)
                if (e[k] < kTombKey && !(last && k == kKeys - 1)) {
                    keys |= 1u << k;
                    if (kBits)
                        out |= (inside(e[k]) ^ 1u) << k;
                }
            edges += __popc(keys);
            if (kBits) {
                const bool u_in = (in >> it) & 1u;
                const uint32_t need = u_in ? out : keys;
                if (!__any_sync(kFull, need))
                    continue;
                const uint32_t own = __shfl_sync(kFull, own_l, it), a = u_in ? root : own;
#pragma unroll
                for (int k = 0; k < kKeys; ++k) {
                    const uint32_t m = __ballot_sync(kFull, (need >> k) & 1u);
                    if ((need >> k) & 1u)
                        pairs[w][held + __popc(m & lanemask_lt())] = make_uint2(a, (out >> k) & 1u ? e[k] : root);
                    held += __popc(m);
                }
                __syncwarp();
                while (held >= 64) {
                    held -= 64;
                    united += 64;
                    ok = unite_pairs(p, &pairs[w][held], 64) && ok;
                }
            } else {
                const uint32_t own = __shfl_sync(kFull, own_l, it);
                bool act[kKeys];
#pragma unroll
                for (int k = 0; k < kKeys; ++k)
                    act[k] = (keys >> k) & 1u;
                if (last) {
                    e[kKeys - 1] = own;
                    act[kKeys - 1] = (live >> it) & 1u;
                }
                ok = group_union<kLanes, kKeys>(p, e, act, 1u << 20) && ok;
            }
        }
    }
    if (kBits && held)
        ok = unite_pairs(p, pairs[w], held) && ok;
    if (!ok)
        *failed = 1;
    count_add(g.st, kCtrWccSlabs, slabs);
    const uint32_t all = __reduce_add_sync(kFull, edges);
    count_add(g.st, kCtrWccEdges, all);
    count_add(g.st, kCtrWccUnited, kBits ? united + held : all);
}

namespace mk {

template <bool kSet>
static cudaError_t launch_static(const GView &g, uint32_t *p, uint32_t *label, uint32_t *bits, uint32_t *giant,
                                 int *failed, cudaStream_t s, int *launches)
{
    const uint32_t vgrid = grid_for(g.V, 256);
    const size_t bytes = ((size_t)g.V + 31) / 32 * 4;
    // largest bitmap in shared memory, beside 50 KB of pairs
    constexpr size_t kCcBitBytes = 160 << 10;
    // A graph of few slabs is scanned in less time than the sample takes to
    // launch.
    if (g.H < kCcSampleLists) {
        k_uf_init<<<vgrid, 256, 0, s>>>(p, g.V);
        static const uint32_t grid = resident_grid(k_cc_scan<kSet, 0>, kScanThreads);
        k_cc_scan<kSet, 0><<<grid, kScanThreads, 0, s>>>(g, p, nullptr, nullptr, failed);
        *launches += 2;
    } else {
        k_cc_sample<kSet><<<vgrid, 256, 0, s>>>(g, p);
        k_uf_compress<<<vgrid, 256, 0, s>>>(p, g.V, nullptr, nullptr, g.st);
        k_cc_link<kSet><<<grid_for(g.V / kLinkStep + 1, 256), 256, 0, s>>>(g, p);
        k_uf_compress<<<vgrid, 256, 0, s>>>(p, g.V, nullptr, nullptr, g.st);
        k_cc_giant<<<1, 1024, 0, s>>>(p, g.V, giant);
        k_cc_bits<<<vgrid, 256, 0, s>>>(p, g.V, giant, bits);
        if (bytes <= kCcBitBytes) {
            auto k = k_cc_scan<kSet, 1>;
            // (not `bytes`: another thread may be about to launch it for a larger graph)
            cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kCcBitBytes);
            if (e != cudaSuccess)
                return e;
            k<<<num_sms(), kScanThreads, bytes, s>>>(g, p, bits, giant, failed);
        } else {
            k_cc_scan<kSet, 2><<<num_sms(), kScanThreads, 0, s>>>(g, p, bits, giant, failed);
        }
        *launches += 7;
    }
    k_uf_compress<<<vgrid, 256, 0, s>>>(p, g.V, label, failed, g.st);
    *launches += 1;
    return cudaGetLastError();
}

cudaError_t static_components(const GView &g, bool set, uint32_t *p, uint32_t *label, uint32_t *bits, uint32_t *giant,
                              int *failed, cudaStream_t s, int *launches)
{
    return set ? launch_static<true>(g, p, label, bits, giant, failed, s, launches)
               : launch_static<false>(g, p, label, bits, giant, failed, s, launches);
}

} // namespace mk

extern "C" mk_status mk_incr_wcc(mk_graph *g, uint32_t *d_label, void *stream)
{
    if (!g)
        return MK_ERR_INVALID_ARG;
    cudaStream_t s = (cudaStream_t)stream;
    const uint32_t V = g->v.V;
    auto key = std::make_pair((int)kWcc, 0u);
    Consumer *c = nullptr;
    auto it = g->consumers.find(key);
    if (it == g->consumers.end()) {
        c = new Consumer;
        c->kind = kWcc;
        mk_status st = device_alloc(g, (void **)&c->uf, (size_t)V * 4, s);
        if (st == MK_OK)
            st = device_alloc(g, (void **)&c->inv, ((size_t)V + 31) / 32 * 4, s);
        if (st == MK_OK)
            st = device_alloc(g, (void **)&c->counters, kConsumerWords * 4, s);
        if (st != MK_OK) {
            device_free(g, c->uf, (size_t)V * 4, s);
            device_free(g, c->inv, ((size_t)V + 31) / 32 * 4, s);
            device_free(g, c->counters, kConsumerWords * 4, s);
            delete c;
            return st;
        }
        g->consumers[key] = c;
    } else {
        c = it->second;
    }
    // the paper has no decremental WCC: an epoch with deletions recomputes
    const bool incremental = c->epoch == g->epoch && !g->epoch_has_deletes;
    const uint32_t max_hops = g->v.P + 2;
    int *failed = (int *)c->counters;
    MK_CUDA(cudaMemsetAsync(c->counters, 0, 64, s));
    if (!incremental) {
        int launches = 0;
        MK_TRY(timed(g, "wcc_static", s, 0, [&]() {
            return static_components(g->v, false, c->uf, d_label, c->inv, c->counters + 1, failed, s, &launches);
        }));
        g->launches += (uint64_t)launches;
    } else {
        MK_TRY(timed(g, "wcc_hook_updated", s, 1, [&]() {
            if (g->ilog_ok && g->d_ilog) {
                const uint64_t threads = std::max<uint64_t>(g->ilog_bound, 1);
                k_uf_hook_log<<<std::min<uint32_t>(grid_for(threads, 256), num_sms() * 8), 256, 0, s>>>(
                    g->d_state, g->d_ilog, g->ilog_bound, c->uf, failed);
            } else {
                // one 4-lane group per logged list
                const uint64_t threads = std::max<uint64_t>(g->ulog_bound, 1) * 4;
                k_uf_hook<<<std::min<uint32_t>(grid_for(threads, 256), num_sms() * 12), 256, 0, s>>>(
                    g->v, c->uf, max_hops, failed);
            }
            return cudaSuccess;
        }));
        MK_TRY(timed(g, "wcc_compress", s, 1, [&]() {
            k_uf_compress<<<grid_for(V, 256), 256, 0, s>>>(c->uf, V, d_label, failed, g->d_state);
            return cudaSuccess;
        }));
    }
    c->epoch = g->epoch;
    c->seq = g->change_seq;
    return MK_OK;
}
