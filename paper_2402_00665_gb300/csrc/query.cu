// query.cu -- stackless range queries (Algorithm 1) and CSR assembly.
//
// Sphere and box queries take the leaf blocks (packet.cu) unless they are
// many but far apart, and few rays too; what follows is the walk of the nodes
// for the others, for trees from checkpoints (it checks their links) and for
// the tuner's other walk variants. Each thread walks the tree for one query: start at the root (id 0); when
// the predicate holds on an internal node go to its left child, on a leaf
// report it and go to its skip; when it fails go to the skip; stop at the
// sentinel. Every step runs the same code for internal nodes and leaves: a
// 16-byte load (internal: lo + left; point leaf: xyz + index word), a second
// one for internal nodes and box leaves (hi + skip), the box test, and a
// select. A leaf's skip is position k+1, leaf or internal by one bit.
//
// Predicates (closed, FP32, fixed operation order):
//   sphere  e_a = max(lo_a - c_a, c_a - hi_a, 0);
//           d2 = fma(ez, ez, fma(ey, ey, ex*ex)) (each step rounded once);
//           hit iff d2 <= r*r. Every step is monotone in e_a >= 0, so a
//           node's d2 never exceeds the d2 of a primitive inside it: the walk
//           prunes nothing a brute-force scan would report. e_a is computed
//           as c_a - clamp(c_a, lo_a, hi_a), which has the same magnitude
//           because fl(x - y) = -fl(y - x).
//   box     lo_q <= hi_b and lo_b <= hi_q on every axis.
//   ray     the slab test of a segment {origin, tmin, direction, tmax}
//           (see hits(const Ray &...)); many rays are walked by the 256
//           cells of their middles.
//
// Threads take the queries in the order given by QueryArgs::order (the
// queries sorted along a curve through their centres, so that a warp's walks
// visit the same nodes), and write results at the query's own index.
//
// CSR in one walk:
//   collect   each thread walks sorted position i (query q = order[i]; groups
//             of lanes walking together are a tuning option) and writes up
//             to kQueryBufferHits primitive ids, in walk order, into slot q
//             of a scratch array (no shared memory: L1 stays with the tree),
//             and the hit count at q. Slot q rather than slot i: the copy
//             then reads the slots in order (copy 1.86 -> 1.45 ms on 2^25
//             uniform points; the walk's stores are scattered either way).
//   scan      exclusive scan of the counts -> offsets, total (host reads
//             it): one kernel with a bounded look-back, or three for many.
//   copy      in query order: each thread loads one slot of up to 32 hits
//             into registers and sorts it with an odd-even merge network;
//             the warp's 32 lists, adjacent in the CSR, leave through shared
//             memory as one run; lists of 33..64 hits are sorted by the
//             whole warp (two values per lane, shuffles).
//   overflow  hits past the slot go on, during the same walk, to chunks of a
//             shared spill pool; those lists are copied (slot + chunks) to
//             their CSR ranges; only when the pool runs out does a query walk
//             a second time, writing straight into the CSR. A fix-up kernel
//             then sorts every such list, one warp per list (one CTA per list
//             above 1024 hits).
#include <algorithm>
#include <atomic>
#include <cstdlib>
#include <type_traits>

#include "lbvh_internal.cuh"
#include "morton.cuh"
#include "walk.cuh"

namespace lbvh {

namespace {

constexpr int kThreads = 256;

// Algorithm 1. on_leaf(id) is called with the primitive index of every leaf
// that satisfies the predicate, leaves in increasing sorted position. Returns
// false if the walk ran past 2(2n-1) steps or met an id outside the tree (a
// corrupt tree).
template <int kP, typename Q, typename F>
__device__ __forceinline__ bool walk(const TreeView &t, const Q &q, F &&on_leaf) {
    const int ni = (int)t.n - 1;
    const int nodes = 2 * (int)t.n - 1;
    const uint32_t max_steps = 2u * (uint32_t)nodes;
    const float4 *base = t.inodes;  // leaves follow the internal records
    int node = 0;
    uint32_t steps = 0;
    // ids outside [0, nodes) end the loop: the sentinel, one past the last
    // leaf (the last leaf's skip), or a corrupt id (reported below)
    while ((uint32_t)node < (uint32_t)nodes) {
        if (++steps > max_steps) return false;
        const bool leaf = node >= ni;
        const int unit = kP == LBVH_PRIM_BOXES ? 2 * node : (leaf ? node + ni : 2 * node);
        float4 a, b;
        load_node<kP>(base, unit, leaf, a, b);
        const bool hit = hits(q, xyz(a), xyz(b));
        const uint32_t word = __float_as_uint(a.w);
        if (hit && leaf) on_leaf(word & kLeafIndexMask);
        // internal: left child on a hit, else skip; leaf k: position k+1
        node = leaf ? node + 1 - ((word & kLeafSkipInternal) ? ni : 0)
                    : __float_as_int(hit ? a.w : b.w);
    }
    return node == kSentinel || node == nodes;
}

// Algorithm 1 walked by a group of kLanes adjacent lanes together (8, 16 or
// 32): the group stands at one node, every lane tests its own query there,
// and at an internal node the group goes to the left child if any lane's
// predicate holds, else to the skip. Every lane calls on_leaf for each leaf
// its own predicate accepts. The group's walk visits every node that one of
// its lanes' own walks visits (a leaf a lane accepts has all its ancestors
// accepted by that lane, the predicates being monotone), in the same
// pre-order, so each lane reports exactly its own walk's hits, in the same
// order. A step loads one node for the whole group (a broadcast) instead of
// one per lane, and walks the union of the lanes' paths. Lanes without a
// query (active false) walk along and report nothing.
template <int kP, int kLanes, typename Q, typename F>
__device__ __forceinline__ bool walk_group(const TreeView &t, const Q &q, bool active, F &&on_leaf) {
    const int ni = (int)t.n - 1;
    const int nodes = 2 * (int)t.n - 1;
    const uint32_t max_steps = 2u * (uint32_t)nodes;
    const float4 *base = t.inodes;
    const int lane = threadIdx.x & 31;
    const uint32_t gmask =
        kLanes == 32 ? 0xffffffffu : (((1u << kLanes) - 1u) << (lane & ~(kLanes - 1)));
    int node = 0;
    uint32_t steps = 0;
    while ((uint32_t)node < (uint32_t)nodes) {
        if (++steps > max_steps) return false;
        const bool leaf = node >= ni;
        const int unit = kP == LBVH_PRIM_BOXES ? 2 * node : (leaf ? node + ni : 2 * node);
        float4 a, b;
        load_node<kP>(base, unit, leaf, a, b);
        const bool hit = active && hits(q, xyz(a), xyz(b));
        const uint32_t word = __float_as_uint(a.w);
        if (leaf) {
            if (hit) on_leaf(word & kLeafIndexMask);
            node = node + 1 - ((word & kLeafSkipInternal) ? ni : 0);
        } else {
            node = __float_as_int((__ballot_sync(gmask, hit) & gmask) ? a.w : b.w);
        }
    }
    return node == kSentinel || node == nodes;
}

// One query's collecting walk at walk position i (query qi): the first kSlot
// hits go to the slot, later ones to spill chunks. Writes (count, i) and, for
// a long list, its overflow-list entry (tagged when all its hits are in slot
// + chunks).
// kLanes = 0: the thread walks alone (walk); else with its group of kLanes
// lanes (walk_group; every lane of the warp must call this, `has_query`
// false for lanes past the last query).
template <int kQ, int kP, bool kPairs, int kLanes = 0>
__device__ __forceinline__ void collect_walk(const TreeView &t, const QueryArgs &qa, const QueryScratch &qs,
                                             Control *ctl, int64_t i, int64_t qi, bool walk_ok,
                                             bool has_query = true) {
    uint32_t cnt = 0;
    uint32_t cur = kNoChunk;
    if (walk_ok) {
        const auto q = has_query ? QueryOf<kQ>::load(qa, qi) : typename QueryOf<kQ>::type{};
        uint32_t *slot = qs.slots + qi * kSlot;
        // kPairs: hits go to the slot two at a time (one 8-byte store; words
        // past the count are never read). Point trees, one tree: walk 16.19
        // -> 15.87 ms on 2^25 uniform points (held to 32 registers, with an
        // 8-byte spill; 16.00 ms at 40 registers); on box trees it cost more
        // (D3 walk 8.39 -> 8.49 ms at 40 registers).
        uint2 buf = make_uint2(0u, 0u);
        auto keep = [&](uint32_t id) {
            if (cnt < (uint32_t)kSlot) {
                if (!kPairs) {
                    __stcs(slot + cnt, id);
                } else if (cnt & 1u) {
                    buf.y = id;
                    __stcs(reinterpret_cast<uint2 *>(slot + cnt - 1), buf);
                } else {
                    buf.x = id;
                }
            } else {
                spill_put(qs, ctl, qi, cnt, id, cur);
            }
            ++cnt;
        };
        bool ok;
        if constexpr (kLanes == 0 && kQ == LBVH_Q_RAY) {
            // one instruction stream for the warp: the general test if any of its rays has a parallel axis
            if (__any_sync(__activemask(), q.parallel != 0))
                ok = walk<kP>(t, q, keep);
            else
                ok = walk<kP>(t, SlantedRay{q}, keep);
        } else if constexpr (kLanes == 0)
            ok = walk<kP>(t, q, keep);
        else
            ok = walk_group<kP, kLanes>(t, q, has_query, keep);
        if (!has_query) return;
        if (kPairs && cnt < (uint32_t)kSlot && (cnt & 1u)) __stcs(reinterpret_cast<uint2 *>(slot + cnt - 1), buf);
        if (!ok) atomicOr(&ctl->query_flags, kFlagCorrupt);
    }
    if (!has_query) return;
    __stcs(qs.counts + qi, cnt);  // streamed: keep L2 for the tree
    if (cnt > (uint32_t)kSlot)
        qs.overflow_list[atomicAdd(&ctl->overflow_filled, 1u)] =
            (uint32_t)qi | (cur != kSpillFailed ? kSpilledTag : 0u);
}

// The collecting walk with groups of kLanes lanes walking together
// (walk_group); thread i takes walk position i as in collect_kernel.
template <int kQ, int kP, int kLanes>
__global__ void __launch_bounds__(kThreads, 8)
    collect_group_kernel(TreeView t, QueryArgs qa, QueryScratch qs, Control *ctl) {
    const int64_t i = (int64_t)blockIdx.x * kThreads + threadIdx.x;
    const int64_t warp_first = i - (threadIdx.x & 31);
    if (warp_first >= qa.nq) return;  // whole warps leave together
    const bool has = i < qa.nq;
    const bool walk_ok = t.n > 0 && ctl->build_flags == 0;
    collect_walk<kQ, kP, kP == LBVH_PRIM_POINTS, kLanes>(t, qa, qs, ctl, i, has ? query_at<kQ>(qa, i) : 0, walk_ok,
                                                       has);
}

// One thread per walk position: thread i walks position i (query order[i]).
// At most 32 registers (2048 threads per SM): the walk hides its load latency
// with occupancy. Several walks per thread in lock step (K independent loads
// in flight per thread) measured slower on GB300: the walk is bound by L1
// wavefronts (distinct sectors per load), which more walks per thread only
// increase. kT threads per CTA (256 or 512, a tuner choice): the CTAs that
// share an SM's L1 walk kT adjacent queries each, so larger CTAs put more
// neighbouring walks on one SM (D2 walk 15.93 -> 15.66 ms with 512; 1024
// measured slower on D2 and D3).
template <int kQ, int kP, int kT>
__global__ void __launch_bounds__(kT, 2048 / kT)
    collect_kernel(TreeView t, QueryArgs qa, QueryScratch qs, Control *ctl) {
    const int64_t i = (int64_t)blockIdx.x * kT + threadIdx.x;
    if (i >= qa.nq) return;
    const bool walk_ok = t.n > 0 && ctl->build_flags == 0;
    collect_walk<kQ, kP, kP == LBVH_PRIM_POINTS>(t, qa, qs, ctl, i, query_at<kQ>(qa, i), walk_ok);
}

// The queries that packet_kernel left (packets of queries too far apart; list
// entries of 32 walk positions each). A few entries: 8 lanes per query
// through the leaf blocks, 4 queries per warp (2^24 box queries on 2^25 boxes
// leave about 200 entries: Algorithm 1 took 0.29 ms, one long walk after the
// other). Many: Algorithm 1, a warp per entry, the faster one when the GPU is
// full. A fixed grid strides over the list.
constexpr int64_t kLeftFew = 2048;

template <int kQ, int kP>
__global__ void __launch_bounds__(kThreads)
    collect_left_kernel(TreeView t, const float4 *__restrict__ rec, QueryArgs qa, QueryScratch qs, Control *ctl) {
    __shared__ uint32_t s_stack[kThreads / 8][kSparseStack];
    const int64_t count = ctl->sparse_filled;
    const int lane = threadIdx.x & 31;
    const int64_t stride = (int64_t)gridDim.x * (kThreads / 32);
    const int64_t first = ((int64_t)blockIdx.x * kThreads + threadIdx.x) >> 5;
    if (count <= kLeftFew) {
        const Blocks blocks{t.leaves, rec, (int)t.n, pack_leaf_start(t.n)};
        for (int64_t j = first; j < 8 * count; j += stride) {
            const uint2 e = qs.sparse_list[j >> 3];
            const int at = (int)(j & 7) * 4 + (lane >> 3);
            const bool has = (e.y >> at) & 1u;
            const int64_t qi = has ? thread_query(qa, (int64_t)e.x * 32 + at) : 0;
            typename QueryOf<kQ>::type q{};
            if (has) q = QueryOf<kQ>::load(qa, qi);
            sparse_walk<kP>(blocks, s_stack[threadIdx.x >> 3], q, has, qi, qs, ctl);
        }
        return;
    }
    for (int64_t j = first; j < count; j += stride) {
        const uint2 e = qs.sparse_list[j];
        const int64_t i = (int64_t)e.x * 32 + lane;
        if ((e.y >> lane) & 1u)
            collect_walk<kQ, kP, kP == LBVH_PRIM_POINTS>(t, qa, qs, ctl, i, thread_query(qa, i), true);
    }
}

// Batcher's odd-even merge sort of v[0..kN) (kN a power of two), keeping only
// the comparators inside v[0..kAct). Every comparator puts the smaller value
// at the lower index, so padding values ~0u at the top never move and the
// comparators that reach them do nothing: the pruned network sorts kAct
// values (8: 19 comparators, 16: 63, 24: 132, 32: 191; a bitonic network
// over 32 takes 240). Written as templates so that every index is a
// compile-time constant and v stays in registers.
template <int kAct>
__device__ __forceinline__ void compare_swap(uint32_t (&v)[32], int x, int y) {
    if (y < kAct) {
        const uint32_t a = v[x], b = v[y];
        v[x] = min(a, b);
        v[y] = a ^ b ^ v[x];  // the other one; as a second min / max the copy of 2^25 lists takes 1.19 ms, so 1.16
    }
}

// merges the two sorted halves of the elements lo, lo + r, lo + 2r, ... of v[lo, lo + n)
template <int kLo, int kN, int kR, int kAct>
struct OddEvenMerge {
    static __device__ __forceinline__ void run(uint32_t (&v)[32]) {
        constexpr int m = 2 * kR;
        if constexpr (m < kN) {
            OddEvenMerge<kLo, kN, m, kAct>::run(v);
            OddEvenMerge<kLo + kR, kN, m, kAct>::run(v);
#pragma unroll
            for (int i = kLo + kR; i + kR < kLo + kN; i += m) compare_swap<kAct>(v, i, i + kR);
        } else {
            compare_swap<kAct>(v, kLo, kLo + kR);
        }
    }
};

template <int kLo, int kN, int kAct>
struct OddEvenSort {
    static __device__ __forceinline__ void run(uint32_t (&v)[32]) {
        if constexpr (kN > 1) {
            OddEvenSort<kLo, kN / 2, kAct>::run(v);
            OddEvenSort<kLo + kN / 2, kN / 2, kAct>::run(v);
            OddEvenMerge<kLo, kN, 1, kAct>::run(v);
        }
    }
};

template <int kN, int kAct>
__device__ __forceinline__ void merge_sort_net(uint32_t (&v)[32]) {
    OddEvenSort<0, kN, kAct>::run(v);
}

// Ascending bitonic sort of 64 values held by a warp, value e in lane e % 32
// (v0: e < 32, v1: e >= 32). Steps with partner distance 32 compare a lane's
// two values; the others exchange with lane ^ j by shuffle.
__device__ __forceinline__ void warp_sort64(uint32_t &v0, uint32_t &v1) {
    const int lane = threadIdx.x & 31;
#pragma unroll
    for (int k = 2; k <= 64; k <<= 1) {
#pragma unroll
        for (int j = k >> 1; j > 0; j >>= 1) {
            if (j == 32) {  // k == 64: one ascending merge
                const uint32_t lo = min(v0, v1), hi = max(v0, v1);
                v0 = lo;
                v1 = hi;
            } else {
                const bool lower = (lane & j) == 0;
                const uint32_t p0 = __shfl_xor_sync(0xffffffffu, v0, j);
                const uint32_t p1 = __shfl_xor_sync(0xffffffffu, v1, j);
                const bool up0 = (lane & k) == 0, up1 = ((lane + 32) & k) == 0;
                v0 = lower == up0 ? min(v0, p0) : max(v0, p0);
                v1 = lower == up1 ? min(v1, p1) : max(v1, p1);
            }
        }
    }
}

// A warp's 32 lists, none longer than kAct (c hits of this thread, at src):
// loaded, sorted in registers (padded with ~0u) and put one after the other
// into shared memory from place `at` on (this thread's place).
template <int kN, int kAct>
__device__ __forceinline__ void sort_short_lists(const uint4 *src, uint32_t c, uint32_t *flat, uint32_t at) {
    uint32_t v[kRegSort];
#pragma unroll
    for (int j4 = 0; j4 < kAct / 4; ++j4) {
        uint4 w = make_uint4(~0u, ~0u, ~0u, ~0u);
        if (4 * j4 < (int)c) w = src[j4];
        v[4 * j4] = w.x;  // c > 4 j4, or padding already
        v[4 * j4 + 1] = 4 * j4 + 1 < (int)c ? w.y : ~0u;
        v[4 * j4 + 2] = 4 * j4 + 2 < (int)c ? w.z : ~0u;
        v[4 * j4 + 3] = 4 * j4 + 3 < (int)c ? w.w : ~0u;
    }
    merge_sort_net<kN, kAct>(v);
#pragma unroll
    for (int j = 0; j < kAct; ++j)
        if (j < (int)c) flat[at + j] = v[j];
}

// The offsets can be followed and the lists fit the caller's buffer. After a
// wait of the scan has run out, offsets of later tiles and the total are too
// small while earlier ones are not: nothing may be written by them.
__device__ __forceinline__ bool lists_fit(const Control *ctl, unsigned long long capacity) {
    return ctl->total <= capacity && (ctl->query_flags & kFlagTimeout) == 0;
}

// Thread q sorts query q's list in registers if it has at most 32 hits; the
// lists of a warp are adjacent in the CSR, so without a longer one among them
// they go through shared memory as one run and out 32 words per step (2^25
// uniform points, 16 hits: 1.40 -> 1.16 ms; one list per step before, twice the
// steps). Else one list per step with lanes on consecutive hits, and lists of
// 33..64 hits are then sorted and written by the whole warp, one after the
// other; longer ones elsewhere. Five CTAs to an SM: 1.19 ms (2^25 boxes 0.69); the
// four that come without a bound 1.21 (0.72), six 1.53 (spills), three 1.32
// (before compare_swap took its maximum by XOR: now 1.16, 0.68).
__global__ void __launch_bounds__(kThreads, 5)
    copy_kernel(int64_t nq, const uint32_t *__restrict__ counts, const int64_t *__restrict__ offsets,
                const uint32_t *__restrict__ slots, uint32_t *__restrict__ hits,
                unsigned long long capacity, Control *ctl) {
    __shared__ uint32_t s_lists[kThreads / 32][32][kRegSort + 1];
    if (!lists_fit(ctl, capacity)) {  // write nothing
        if (blockIdx.x == 0 && threadIdx.x == 0 && ctl->total > capacity) atomicOr(&ctl->query_flags, kFlagCapacity);
        return;
    }
    const int64_t q = (int64_t)blockIdx.x * kThreads + threadIdx.x;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    uint32_t c = 0, mid = 0;
    bool longer = false;
    int64_t dst = 0, pos = 0;
    if (q < nq) {
        const uint32_t cq = counts[q];
        c = cq > (uint32_t)kRegSort ? 0u : cq;
        longer = cq > (uint32_t)kRegSort;
        mid = longer && cq <= (uint32_t)kSlot ? cq : 0u;  // longer still: the overflow lists
        pos = q;
        dst = offsets[q];
    }
    const uint4 *src = reinterpret_cast<const uint4 *>(slots + pos * kSlot);
    const uint32_t cmax = __reduce_max_sync(kFull, c);
    if (!__any_sync(kFull, longer)) {
        if (cmax == 0) return;
        const int64_t first = __shfl_sync(kFull, dst, 0);
        uint32_t *flat = &s_lists[warp][0][0];
        const uint32_t at = q < nq ? (uint32_t)(dst - first) : 0u;
        const int total = (int)__reduce_max_sync(kFull, at + c);
        if (cmax > 24) sort_short_lists<32, 32>(src, c, flat, at);
        else if (cmax > 16) sort_short_lists<32, 24>(src, c, flat, at);
        else if (cmax > 8) sort_short_lists<16, 16>(src, c, flat, at);
        else sort_short_lists<8, 8>(src, c, flat, at);
        __syncwarp();
        for (int i = lane; i < total; i += 32) hits[first + i] = flat[i];
        return;
    }
    uint32_t mids = __ballot_sync(kFull, mid != 0);
    if (cmax == 0 && mids == 0) return;
    {
        uint32_t *own = s_lists[warp][lane];
        sort_short_lists<32, 32>(src, c, own, 0u);
    }
    __syncwarp();
    for (int s = 0; s < 32; ++s) {
        const uint32_t cs = __shfl_sync(0xffffffffu, c, s);
        const int64_t ds = __shfl_sync(0xffffffffu, dst, s);
        if ((uint32_t)lane < cs) hits[ds + lane] = s_lists[warp][s][lane];
    }
    while (mids) {
        const int s = __ffs(mids) - 1;
        mids &= mids - 1;
        const uint32_t m = __shfl_sync(0xffffffffu, mid, s);
        const int64_t ps = __shfl_sync(0xffffffffu, pos, s);
        const int64_t ds = __shfl_sync(0xffffffffu, dst, s);
        const uint32_t *slot = slots + ps * kSlot;
        uint32_t v0 = (uint32_t)lane < m ? slot[lane] : ~0u;
        uint32_t v1 = (uint32_t)lane + 32 < m ? slot[lane + 32] : ~0u;
        warp_sort64(v0, v1);
        if ((uint32_t)lane < m) hits[ds + lane] = v0;
        if ((uint32_t)lane + 32 < m) hits[ds + lane + 32] = v1;
    }
}

// Second walk for the overflow list: hits go straight to the CSR in walk
// order (sorted afterwards by the list sorts).
template <int kQ, int kP>
__global__ void __launch_bounds__(kThreads)
    overflow_walk_kernel(TreeView t, QueryArgs qa, const uint32_t *__restrict__ list, uint32_t count,
                         const int64_t *__restrict__ offsets, uint32_t *__restrict__ hits) {
    const int64_t j = (int64_t)blockIdx.x * kThreads + threadIdx.x;
    if (j >= count) return;
    const uint32_t e = list[j];
    if (e & kSpilledTag) return;  // its hits are in its slot and spill chunks
    const int64_t qi = e;
    const int64_t base = offsets[qi];
    const int64_t total = offsets[qi + 1] - base;
    const auto q = QueryOf<kQ>::load(qa, qi);
    int64_t c = 0;
    walk<kP>(t, q, [&](uint32_t id) {
        if (c < total) hits[base + c] = id;
        ++c;
    });
}

// ---------------------------------------------------------------- scan
constexpr int kScanThreads = 256;
constexpr int kScanItems = 16;
constexpr int kScanTile = kScanThreads * kScanItems;

__device__ __forceinline__ int64_t block_scan_exclusive(int64_t v, int64_t *s_warp, int64_t &total) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    int64_t x = v;
    for (int off = 1; off < 32; off <<= 1) {
        const int64_t y = __shfl_up_sync(0xffffffffu, x, off);
        if (lane >= off) x += y;
    }
    if (lane == 31) s_warp[warp] = x;
    __syncthreads();
    int64_t before = 0, all = 0;
    for (int w = 0; w < kScanThreads / 32; ++w) {
        if (w < warp) before += s_warp[w];
        all += s_warp[w];
    }
    __syncthreads();
    total = all;
    return before + x - v;
}

// One pass over the counts by decoupled look-back: tiles are taken by ticket
// (so every tile one waits for is running), a tile publishes its sum, then the
// sum of all tiles up to it. state words (zero beforehand, one per tile): bits
// 63:62 = 0 none, 1 the tile's sum, 2 the sum up to the tile. With one tile
// there is nothing to wait for and neither the words nor the ticket are used.
// For up to kScanOnePass tiles per SM, where a tile seldom waits (one launch /
// three below, us: 1,000 counts 5.6 / 12.6; 10^5 9.2 / 14.3; 10^6 13.3 / 16.3;
// 2 10^6 19.4 / 18.3; 4 10^6 33 / 22; 2^25 203 / 121).
// Loads and stores run across the block (thread t at t, t + 256, ...); each
// thread scans kScanItems consecutive counts, which it reads from and writes
// back to shared memory (rows padded by one element against bank conflicts).
constexpr int64_t kScanOnePass = 2;  // tiles per SM
constexpr unsigned long long kScanSum = 1ull << 62, kScanPrefix = 2ull << 62, kScanValue = kScanSum - 1ull;
constexpr unsigned long long kScanWaitNs = 1000000000ull;  // a wait gives up after about a second
constexpr uint32_t kScanSpins = 1u << 26;                  // or after this many polls, whatever the clock says

__device__ __forceinline__ unsigned long long scan_word(const unsigned long long *p) {
    unsigned long long v;
    asm volatile("ld.relaxed.gpu.global.u64 %0, [%1];" : "=l"(v) : "l"(p) : "memory");
    return v;
}
__device__ __forceinline__ void set_scan_word(unsigned long long *p, unsigned long long v) {
    asm volatile("st.relaxed.gpu.global.u64 [%0], %1;" ::"l"(p), "l"(v) : "memory");
}

// The sum of all tiles before `tile` (> 0), by one warp.
__device__ __forceinline__ int64_t scan_look_back(const unsigned long long *state, int64_t tile, Control *ctl) {
    const int lane = threadIdx.x & 31;
    int64_t sum = 0;
    for (int64_t last = tile - 1;; last -= 32) {
        const int64_t at = last - lane;
        unsigned long long v = at >= 0 ? scan_word(state + at) : kScanPrefix;
        if (__any_sync(kFull, (v >> 62) == 0)) {
            unsigned long long t0, now;
            asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t0));
            for (uint32_t spins = 0; __any_sync(kFull, (v >> 62) == 0); ++spins) {
                if ((v >> 62) == 0) v = scan_word(state + at);
                asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(now));
                if (spins > kScanSpins || now - t0 > kScanWaitNs) {
                    if ((v >> 62) == 0) {
                        atomicOr(&ctl->query_flags, kFlagTimeout);
                        v = kScanPrefix;  // give up: results are flagged invalid
                    }
                }
            }
        }
        const uint32_t full = __ballot_sync(kFull, (v >> 62) == 2);
        const int stop = full ? __ffs(full) - 1 : 31;
        int64_t x = lane <= stop ? (int64_t)(v & kScanValue) : 0;
        for (int off = 16; off > 0; off >>= 1) x += __shfl_xor_sync(kFull, x, off);
        sum += x;
        if (full) return sum;
    }
}

__global__ void __launch_bounds__(kScanThreads)
    scan_kernel(const uint32_t *__restrict__ counts, int64_t nq, unsigned long long *state, int64_t *__restrict__ offsets,
                Control *ctl, int64_t hold_tile) {
    constexpr int kRow = kScanItems + 1;
    __shared__ int64_t s_warp[kScanThreads / 32];
    __shared__ int64_t s_o[kScanThreads * kRow];  // the offsets; first the counts (the scan's barriers
                                                  // separate the last read of a count from the first offset)
    __shared__ int64_t s_before;
    __shared__ uint32_t s_tile;
    uint32_t *s_c = reinterpret_cast<uint32_t *>(s_o);
    const bool alone = gridDim.x == 1;
    if (!alone) {
        if (threadIdx.x == 0) s_tile = atomicAdd(&ctl->scan_ticket, 1u);
        __syncthreads();
    }
    const int64_t tile = alone ? 0 : s_tile;
    const int64_t base = tile * kScanTile;
#pragma unroll
    for (int j = 0; j < kScanItems; ++j) {
        const int p = j * kScanThreads + threadIdx.x;
        const int64_t i = base + p;
        s_c[(p / kScanItems) * kRow + p % kScanItems] = i < nq ? counts[i] : 0u;
    }
    __syncthreads();
    uint32_t c[kScanItems];
    int64_t sum = 0;
#pragma unroll
    for (int j = 0; j < kScanItems; ++j) {
        c[j] = s_c[threadIdx.x * kRow + j];
        sum += c[j];
    }
    int64_t total;
    int64_t run = block_scan_exclusive(sum, s_warp, total);
    if (threadIdx.x < 32) {
        const bool publish = !alone && threadIdx.x == 0 && tile != hold_tile;
        if (publish)
            set_scan_word(state + tile, (tile == 0 ? kScanPrefix : kScanSum) | (unsigned long long)total);
        const int64_t before = tile == 0 ? 0 : scan_look_back(state, tile, ctl);
        if (threadIdx.x == 0) {
            if (publish && tile > 0) set_scan_word(state + tile, kScanPrefix | (unsigned long long)(before + total));
            s_before = before;
            if (base + kScanTile >= nq) {  // the last tile
                offsets[nq] = before + total;
                ctl->total = (unsigned long long)(before + total);
            }
        }
    }
    __syncthreads();
    run += s_before;
#pragma unroll
    for (int j = 0; j < kScanItems; ++j) {
        s_o[threadIdx.x * kRow + j] = run;
        run += c[j];
    }
    __syncthreads();
#pragma unroll
    for (int j = 0; j < kScanItems; ++j) {
        const int p = j * kScanThreads + threadIdx.x;
        const int64_t i = base + p;
        if (i < nq) offsets[i] = s_o[(p / kScanItems) * kRow + p % kScanItems];
    }
}

// More tiles than run at once: reduce, scan of the sums, apply.
__global__ void __launch_bounds__(kScanThreads)
    scan_reduce_kernel(const uint32_t *__restrict__ counts, int64_t nq, int64_t *tile_sums) {
    __shared__ int64_t s_warp[kScanThreads / 32];
    const int64_t base = (int64_t)blockIdx.x * kScanTile;
    int64_t sum = 0;
    for (int j = 0; j < kScanItems; ++j) {
        const int64_t i = base + j * kScanThreads + threadIdx.x;
        if (i < nq) sum += counts[i];
    }
    int64_t total;
    block_scan_exclusive(sum, s_warp, total);
    if (threadIdx.x == 0) tile_sums[blockIdx.x] = total;
}

__global__ void __launch_bounds__(kScanThreads)
    scan_tiles_kernel(int64_t *tile_sums, int64_t tiles, int64_t *offsets, int64_t nq,
                      unsigned long long *total_out) {
    __shared__ int64_t s_warp[kScanThreads / 32];
    int64_t carry = 0;
    for (int64_t base = 0; base < tiles; base += kScanThreads) {
        const int64_t i = base + threadIdx.x;
        const int64_t v = i < tiles ? tile_sums[i] : 0;
        int64_t total;
        const int64_t ex = block_scan_exclusive(v, s_warp, total);
        if (i < tiles) tile_sums[i] = carry + ex;
        carry += total;
    }
    if (threadIdx.x == 0) {
        offsets[nq] = carry;
        *total_out = (unsigned long long)carry;
    }
}

// Loads and stores run across the block (thread t at t, t + 256, ...); each
// thread scans kScanItems consecutive counts, which it reads from and writes
// back to shared memory (rows padded by one element against bank conflicts).
__global__ void __launch_bounds__(kScanThreads)
    scan_apply_kernel(const uint32_t *__restrict__ counts, int64_t nq,
                      const int64_t *__restrict__ tile_sums, int64_t *__restrict__ offsets) {
    constexpr int kRow = kScanItems + 1;
    __shared__ int64_t s_warp[kScanThreads / 32];
    __shared__ int64_t s_o[kScanThreads * kRow];  // the offsets; first the counts (the scan's barriers
                                                  // separate the last read of a count from the first offset)
    uint32_t *s_c = reinterpret_cast<uint32_t *>(s_o);
    const int64_t base = (int64_t)blockIdx.x * kScanTile;
#pragma unroll
    for (int j = 0; j < kScanItems; ++j) {
        const int p = j * kScanThreads + threadIdx.x;
        const int64_t i = base + p;
        s_c[(p / kScanItems) * kRow + p % kScanItems] = i < nq ? counts[i] : 0u;
    }
    __syncthreads();
    uint32_t c[kScanItems];
    int64_t sum = 0;
#pragma unroll
    for (int j = 0; j < kScanItems; ++j) {
        c[j] = s_c[threadIdx.x * kRow + j];
        sum += c[j];
    }
    int64_t total;
    int64_t run = tile_sums[blockIdx.x] + block_scan_exclusive(sum, s_warp, total);
#pragma unroll
    for (int j = 0; j < kScanItems; ++j) {
        s_o[threadIdx.x * kRow + j] = run;
        run += c[j];
    }
    __syncthreads();
#pragma unroll
    for (int j = 0; j < kScanItems; ++j) {
        const int p = j * kScanThreads + threadIdx.x;
        const int64_t i = base + p;
        if (i < nq) offsets[i] = s_o[(p / kScanItems) * kRow + p % kScanItems];
    }
}

// ---------------------------------------------------------------- fix-up sort
constexpr int kFixThreads = 512;
constexpr int kFixSmem = 8192;

__device__ __forceinline__ void order_pair(uint32_t *a, int64_t lo, int64_t hi) {
    const uint32_t x = a[lo], y = a[hi];
    if (x > y) {
        a[lo] = y;
        a[hi] = x;
    }
}

// Bitonic sorting network in its one-direction form: every comparator puts
// the smaller value at the lower index (the first step of each merge pairs i
// with the mirror position in its block, later steps pair i with i + j).
// Positions >= m act as +infinity and their comparators are skipped, which
// leaves the network correct for any m.
__device__ void bitonic_sort(uint32_t *a, int64_t m) {
    int64_t pow2 = 1;
    while (pow2 < m) pow2 <<= 1;
    for (int64_t k = 2; k <= pow2; k <<= 1) {
        const int64_t half = k >> 1;
        for (int64_t i = threadIdx.x; i < pow2 / 2; i += blockDim.x) {
            const int64_t blk = i / half, off = i % half;
            const int64_t lo = blk * k + off, hi = blk * k + k - 1 - off;
            if (hi < m) order_pair(a, lo, hi);
        }
        __syncthreads();
        for (int64_t j = k >> 2; j >= 1; j >>= 1) {
            for (int64_t i = threadIdx.x; i < pow2 / 2; i += blockDim.x) {
                const int64_t blk = i / j, off = i % j;
                const int64_t lo = blk * 2 * j + off, hi = lo + j;
                if (hi < m) order_pair(a, lo, hi);
            }
            __syncthreads();
        }
    }
}

// One warp per overflow list (the common case: a few dozen to a few hundred
// hits): the warp loads the list into its own shared-memory region, runs the
// network with __syncwarp between steps and writes it back. Lists longer than
// kWarpSortMax go to a second list (kept in the then unused slot buffer) for
// sort_big_lists_kernel. Both kernels stride over counts held on the device
// and write nothing when the hits did not fit the caller's buffer.
constexpr int kWarpSortMax = 1024;
constexpr int kSortWarps = kThreads / 32;

__device__ void warp_bitonic_sort(uint32_t *a, int m) {
    const int lane = threadIdx.x & 31;
    int lg = 0;
    while ((1 << lg) < m) ++lg;
    const int pairs = (1 << lg) >> 1;
    for (int lk = 1; lk <= lg; ++lk) {
        // first step of the merge of blocks of 2^lk: i pairs with its mirror
        const int lh = lk - 1;
        for (int i = lane; i < pairs; i += 32) {
            const int blk = i >> lh, off = i & ((1 << lh) - 1);
            const int lo = (blk << lk) + off, hi = (blk << lk) + (1 << lk) - 1 - off;
            if (hi < m) order_pair(a, lo, hi);
        }
        __syncwarp();
        for (int lj = lk - 2; lj >= 0; --lj) {
            for (int i = lane; i < pairs; i += 32) {
                const int blk = i >> lj, off = i & ((1 << lj) - 1);
                const int lo = (blk << (lj + 1)) + off, hi = lo + (1 << lj);
                if (hi < m) order_pair(a, lo, hi);
            }
            __syncwarp();
        }
    }
}

__global__ void __launch_bounds__(kThreads)
    warp_sort_lists_kernel(const int64_t *__restrict__ offsets, uint32_t *hits,
                           const uint32_t *__restrict__ list, uint32_t *__restrict__ big_list, Control *ctl,
                           unsigned long long capacity) {
    __shared__ uint32_t s[kSortWarps][kWarpSortMax];
    if (!lists_fit(ctl, capacity)) return;
    const uint32_t count = ctl->overflow_filled;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    uint32_t *a = s[warp];
    for (int64_t j = (int64_t)blockIdx.x * kSortWarps + warp; j < count; j += (int64_t)gridDim.x * kSortWarps) {
        const uint32_t q = list[j] & ~kSpilledTag;
        const int64_t base = offsets[q];
        const int64_t m = offsets[q + 1] - base;
        if (m > kWarpSortMax) {
            if (lane == 0) big_list[atomicAdd(&ctl->overflow_big, 1u)] = q;
            continue;
        }
        uint32_t *seg = hits + base;
        for (int i = lane; i < m; i += 32) a[i] = seg[i];
        __syncwarp();
        warp_bitonic_sort(a, (int)m);
        for (int i = lane; i < m; i += 32) seg[i] = a[i];
        __syncwarp();
    }
}

__global__ void __launch_bounds__(kFixThreads)
    sort_big_lists_kernel(const int64_t *__restrict__ offsets, uint32_t *hits,
                          const uint32_t *__restrict__ big_list, const Control *ctl,
                          unsigned long long capacity) {
    __shared__ uint32_t s[kFixSmem];
    if (!lists_fit(ctl, capacity)) return;
    const uint32_t count = ctl->overflow_big;
    for (uint32_t j = blockIdx.x; j < count; j += gridDim.x) {
        const uint32_t q = big_list[j];
        const int64_t base = offsets[q];
        const int64_t m = offsets[q + 1] - base;
        uint32_t *seg = hits + base;
        if (m <= kFixSmem) {
            for (int64_t i = threadIdx.x; i < m; i += blockDim.x) s[i] = seg[i];
            __syncthreads();
            bitonic_sort(s, m);
            for (int64_t i = threadIdx.x; i < m; i += blockDim.x) seg[i] = s[i];
        } else {
            bitonic_sort(seg, m);  // in global memory; one CTA owns the list
        }
        __syncthreads();
    }
}

// Lists whose hits past the slot all went to spill chunks: one warp per list
// copies the slot and then each chunk of its chain to the list's CSR range
// (in walk order; the list sorts follow).
__global__ void __launch_bounds__(kThreads)
    spill_gather_kernel(QueryScratch qs, const int64_t *__restrict__ offsets, uint32_t *__restrict__ hits,
                        const Control *ctl, unsigned long long capacity) {
    if (!lists_fit(ctl, capacity)) return;
    const uint32_t count = ctl->overflow_filled;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    constexpr int kWarps = kThreads / 32;
    for (int64_t j = (int64_t)blockIdx.x * kWarps + warp; j < count; j += (int64_t)gridDim.x * kWarps) {
        const uint32_t e = qs.overflow_list[j];
        if (!(e & kSpilledTag)) continue;  // walks a second time instead
        const uint32_t q = e & ~kSpilledTag;
        const int64_t base = offsets[q];
        const int64_t m = offsets[q + 1] - base;
        uint32_t *dst = hits + base;
        const uint32_t *slot = qs.slots + (int64_t)q * kSlot;
        for (int k = lane; k < kSlot; k += 32) dst[k] = slot[k];
        int64_t done = kSlot;
        uint32_t c = qs.spill_head[q];
        while (done < m) {
            if (c >= qs.spill_chunks) break;  // cannot happen for a tagged list; guards the reads
            const uint32_t *chunk = qs.spill + (int64_t)c * kSpillChunkWords;
            const int64_t take = min((int64_t)(kSpillChunkWords - 1), m - done);
            for (int k = lane; k < take; k += 32) dst[done + k] = chunk[1 + k];
            done += take;
            c = chunk[0];
        }
    }
}

// ---- batches: the same walk, on the tree of the query's instance

template <int kQ, int kP>
__global__ void __launch_bounds__(kThreads, 8)  // at most 32 registers: full occupancy for the walk
    batch_collect_kernel(const float4 *__restrict__ nodes, BatchTables bt, QueryArgs qa, QueryScratch qs,
                         Control *ctl) {
    const int64_t i = (int64_t)blockIdx.x * kThreads + threadIdx.x;
    if (i >= qa.nq) return;
    const int64_t qi = thread_query(qa, i);
    const int b = instance_of(bt.query_off, bt.count, qi);
    const int64_t n = bt.prim_off[b + 1] - bt.prim_off[b];
    const TreeView t{nodes + bt.node_start[b], nullptr, n, kP};
    collect_walk<kQ, kP, false>(t, qa, qs, ctl, i, qi, n > 0 && ctl->build_flags == 0);
}

template <int kQ, int kP>
__global__ void __launch_bounds__(kThreads, 8)
    batch_collect_left_kernel(const float4 *__restrict__ nodes, BatchTables bt, QueryArgs qa, QueryScratch qs,
                              Control *ctl) {
    const int64_t count = ctl->sparse_filled;
    const int lane = threadIdx.x & 31;
    const int64_t stride = (int64_t)gridDim.x * (kThreads / 32);
    for (int64_t j = ((int64_t)blockIdx.x * kThreads + threadIdx.x) >> 5; j < count; j += stride) {
        const uint2 e = qs.sparse_list[j];
        if (!((e.y >> lane) & 1u)) continue;
        const int64_t i = (int64_t)e.x * 32 + lane, qi = thread_query(qa, i);
        const int b = instance_of(bt.query_off, bt.count, qi);
        const int64_t n = bt.prim_off[b + 1] - bt.prim_off[b];
        const TreeView t{nodes + bt.node_start[b], nullptr, n, kP};
        collect_walk<kQ, kP, false>(t, qa, qs, ctl, i, qi, n > 0);
    }
}

// Overflow lists whose number is known only on the device: a fixed grid
// strides over them.
template <int kQ, int kP>
__global__ void __launch_bounds__(kThreads)
    batch_overflow_kernel(const float4 *__restrict__ nodes, BatchTables bt, QueryArgs qa,
                          const uint32_t *__restrict__ list, const Control *ctl,
                          const int64_t *__restrict__ offsets, uint32_t *__restrict__ hits,
                          unsigned long long capacity) {
    if (!lists_fit(ctl, capacity)) return;
    const uint32_t count = ctl->overflow_filled;
    for (int64_t j = (int64_t)blockIdx.x * kThreads + threadIdx.x; j < count; j += (int64_t)gridDim.x * kThreads) {
        const uint32_t e = list[j];
        if (e & kSpilledTag) continue;  // its hits are in its slot and spill chunks
        const int64_t qi = e;
        const int b = instance_of(bt.query_off, bt.count, qi);
        const int64_t n = bt.prim_off[b + 1] - bt.prim_off[b];
        const TreeView t{nodes + bt.node_start[b], nullptr, n, kP};
        const int64_t base = offsets[qi];
        const int64_t total = offsets[qi + 1] - base;
        const auto q = QueryOf<kQ>::load(qa, qi);
        int64_t c = 0;
        walk<kP>(t, q, [&](uint32_t id) {
            if (c < total) hits[base + c] = id;
            ++c;
        });
    }
}

// ---- walk statistics

// Algorithm 1 for every query, counting the leaves and internal nodes it
// visits (no hits are kept): the walk's work per query, for measurement.
template <int kQ, int kP>
__global__ void __launch_bounds__(kThreads)
    visits_kernel(TreeView t, QueryArgs qa, unsigned long long *counts, Control *ctl) {
    const int64_t i = (int64_t)blockIdx.x * kThreads + threadIdx.x;
    uint32_t leaves = 0, internal = 0;
    if (i < qa.nq && t.n > 0 && ctl->build_flags == 0) {
        const auto q = QueryOf<kQ>::load(qa, query_at<kQ>(qa, i));
        const int ni = (int)t.n - 1;
        const int nodes = 2 * (int)t.n - 1;
        const uint32_t max_steps = 2u * (uint32_t)nodes;
        int node = 0;
        while ((uint32_t)node < (uint32_t)nodes && leaves + internal < max_steps) {
            const bool leaf = node >= ni;
            const int unit = kP == LBVH_PRIM_BOXES ? 2 * node : (leaf ? node + ni : 2 * node);
            float4 a, b;
            load_node<kP>(t.inodes, unit, leaf, a, b);
            const bool hit = hits(q, xyz(a), xyz(b));
            const uint32_t word = __float_as_uint(a.w);
            leaves += leaf;
            internal += !leaf;
            node = leaf ? node + 1 - ((word & kLeafSkipInternal) ? ni : 0) : __float_as_int(hit ? a.w : b.w);
        }
    }
    // one add per warp
    for (int off = 16; off > 0; off >>= 1) {
        leaves += __shfl_xor_sync(0xffffffffu, leaves, off);
        internal += __shfl_xor_sync(0xffffffffu, internal, off);
    }
    if ((threadIdx.x & 31) == 0) {
        atomicAdd(counts, (unsigned long long)leaves);
        atomicAdd(counts + 1, (unsigned long long)internal);
    }
}

}  // namespace

template <typename F>
void dispatch_kinds(int qkind, int pkind, F &&f) {
    if (qkind == LBVH_Q_RAY) {
        if (pkind == LBVH_PRIM_POINTS)
            f(std::integral_constant<int, LBVH_Q_RAY>{}, std::integral_constant<int, LBVH_PRIM_POINTS>{});
        else
            f(std::integral_constant<int, LBVH_Q_RAY>{}, std::integral_constant<int, LBVH_PRIM_BOXES>{});
    } else if (qkind == LBVH_Q_SPHERE) {
        if (pkind == LBVH_PRIM_POINTS)
            f(std::integral_constant<int, LBVH_Q_SPHERE>{}, std::integral_constant<int, LBVH_PRIM_POINTS>{});
        else
            f(std::integral_constant<int, LBVH_Q_SPHERE>{}, std::integral_constant<int, LBVH_PRIM_BOXES>{});
    } else {
        if (pkind == LBVH_PRIM_POINTS)
            f(std::integral_constant<int, LBVH_Q_BOX>{}, std::integral_constant<int, LBVH_PRIM_POINTS>{});
        else
            f(std::integral_constant<int, LBVH_Q_BOX>{}, std::integral_constant<int, LBVH_PRIM_BOXES>{});
    }
}

void launch_query_collect(const TreeView &t, const QueryArgs &q, const QueryScratch &qs, Control *ctl,
                          cudaStream_t s) {
    if (q.nq <= 0) return;
    const unsigned blocks = (unsigned)((q.nq + kThreads - 1) / kThreads);
    dispatch_kinds(q.qkind, t.kind, [&](auto qk, auto pk) {
        constexpr int Q = decltype(qk)::value, P = decltype(pk)::value;
        switch (q.walk) {
        case kWalkGroup8: collect_group_kernel<Q, P, 8><<<blocks, kThreads, 0, s>>>(t, q, qs, ctl); break;
        case kWalkGroup16: collect_group_kernel<Q, P, 16><<<blocks, kThreads, 0, s>>>(t, q, qs, ctl); break;
        case kWalkGroup32: collect_group_kernel<Q, P, 32><<<blocks, kThreads, 0, s>>>(t, q, qs, ctl); break;
        case kWalkThread512:
            collect_kernel<Q, P, 512><<<(unsigned)((q.nq + 511) / 512), 512, 0, s>>>(t, q, qs, ctl);
            break;
        default: collect_kernel<Q, P, kThreads><<<blocks, kThreads, 0, s>>>(t, q, qs, ctl); break;
        }
    });
    count_launches(1);
}

void launch_query_collect_left(const TreeView &t, const float4 *rec, const QueryArgs &q, const QueryScratch &qs,
                               Control *ctl, cudaStream_t s) {
    const unsigned blocks =
        (unsigned)std::min<int64_t>((q.nq + kThreads - 1) / kThreads, (int64_t)device_sm_count() * 8);
    dispatch_kinds(q.qkind, t.kind, [&](auto qk, auto pk) {
        collect_left_kernel<decltype(qk)::value, decltype(pk)::value><<<blocks, kThreads, 0, s>>>(t, rec, q, qs, ctl);
    });
    count_launches(1);
}

void launch_query_copy_checked(const QueryArgs &q, const QueryScratch &qs, const int64_t *offsets,
                               uint32_t *hits, unsigned long long capacity, Control *ctl, cudaStream_t s) {
    if (q.nq <= 0) return;
    const unsigned blocks = (unsigned)((q.nq + kThreads - 1) / kThreads);
    copy_kernel<<<blocks, kThreads, 0, s>>>(q.nq, qs.counts, offsets, qs.slots, hits, capacity, ctl);
    count_launches(1);
}

void launch_query_copy(const QueryArgs &q, const QueryScratch &qs, const int64_t *offsets,
                       uint32_t *hits, Control *ctl, cudaStream_t s) {
    launch_query_copy_checked(q, qs, offsets, hits, ~0ull, ctl, s);
}

// Sorts the overflow lists: warps for the lists, CTAs for the long ones.
// `bound`: an upper bound of the overflow count (sizes the warp kernel's grid).
// First copies the spilled lists (slot + chunks) to their CSR ranges; the
// big-list sort then reuses the slot buffer, which nothing reads any more.
static void launch_sort_lists(const QueryScratch &qs, uint64_t bound, const int64_t *offsets, uint32_t *hits,
                              unsigned long long capacity, Control *ctl, cudaStream_t s) {
    const uint64_t want = (bound + kSortWarps - 1) / kSortWarps;
    const uint64_t cap = (uint64_t)device_sm_count() * 8;
    const unsigned blocks = (unsigned)std::max<uint64_t>(1, std::min(want, cap));
    spill_gather_kernel<<<blocks, kThreads, 0, s>>>(qs, offsets, hits, ctl, capacity);
    warp_sort_lists_kernel<<<blocks, kThreads, 0, s>>>(offsets, hits, qs.overflow_list, qs.slots, ctl, capacity);
    sort_big_lists_kernel<<<(unsigned)device_sm_count(), kFixThreads, 0, s>>>(offsets, hits, qs.slots, ctl,
                                                                              capacity);
    count_launches(3);
}

void launch_query_overflow(const TreeView &t, const QueryArgs &q, const QueryScratch &qs,
                           uint32_t count, const int64_t *offsets, uint32_t *hits, Control *ctl,
                           cudaStream_t s) {
    if (count == 0) return;
    const unsigned blocks = (unsigned)((count + kThreads - 1) / kThreads);
    dispatch_kinds(q.qkind, t.kind, [&](auto qk, auto pk) {
        overflow_walk_kernel<decltype(qk)::value, decltype(pk)::value><<<blocks, kThreads, 0, s>>>(
            t, q, qs.overflow_list, count, offsets, hits);
    });
    launch_sort_lists(qs, count, offsets, hits, ~0ull, ctl, s);
    count_launches(1);
}

void launch_batch_collect(const float4 *nodes, int kind, const BatchTables &bt, const QueryArgs &q,
                          const QueryScratch &qs, Control *ctl, cudaStream_t s) {
    if (q.nq <= 0) return;
    const unsigned blocks = (unsigned)((q.nq + kThreads - 1) / kThreads);
    dispatch_kinds(q.qkind, kind, [&](auto qk, auto pk) {
        batch_collect_kernel<decltype(qk)::value, decltype(pk)::value><<<blocks, kThreads, 0, s>>>(nodes, bt, q, qs,
                                                                                                    ctl);
    });
    count_launches(1);
}

void launch_batch_collect_left(const float4 *nodes, int kind, const BatchTables &bt, const QueryArgs &q,
                               const QueryScratch &qs, Control *ctl, cudaStream_t s) {
    const unsigned blocks =
        (unsigned)std::min<int64_t>((q.nq + kThreads - 1) / kThreads, (int64_t)device_sm_count() * 8);
    dispatch_kinds(q.qkind, kind, [&](auto qk, auto pk) {
        batch_collect_left_kernel<decltype(qk)::value, decltype(pk)::value><<<blocks, kThreads, 0, s>>>(nodes, bt, q, qs,
                                                                                                        ctl);
    });
    count_launches(1);
}

void launch_batch_overflow(const float4 *nodes, int kind, const BatchTables &bt, const QueryArgs &q,
                           const QueryScratch &qs, Control *ctl, const int64_t *offsets, uint32_t *hits,
                           unsigned long long capacity, cudaStream_t s) {
    if (q.nq <= 0) return;
    const unsigned blocks = (unsigned)device_sm_count() * 8;
    dispatch_kinds(q.qkind, kind, [&](auto qk, auto pk) {
        batch_overflow_kernel<decltype(qk)::value, decltype(pk)::value><<<blocks, kThreads, 0, s>>>(
            nodes, bt, q, qs.overflow_list, ctl, offsets, hits, capacity);
    });
    count_launches(1);
    launch_sort_lists(qs, (uint64_t)q.nq, offsets, hits, capacity, ctl, s);
}

void launch_visits(const TreeView &t, const QueryArgs &q, unsigned long long *counts, Control *ctl, cudaStream_t s) {
    if (q.nq <= 0) return;
    const unsigned blocks = (unsigned)((q.nq + kThreads - 1) / kThreads);
    dispatch_kinds(q.qkind, t.kind, [&](auto qk, auto pk) {
        visits_kernel<decltype(qk)::value, decltype(pk)::value><<<blocks, kThreads, 0, s>>>(t, q, counts, ctl);
    });
    count_launches(1);
}

int64_t scan_tile_count(int64_t nq) { return (nq + kScanTile - 1) / kScanTile; }

namespace {
__global__ void __launch_bounds__(kThreads) offsets_add_kernel(int64_t *off, int64_t n, int64_t base) {
    const int64_t i = (int64_t)blockIdx.x * kThreads + threadIdx.x;
    if (i < n) off[i] += base;
}
}  // namespace

void launch_offsets_add(int64_t *offsets, int64_t n, int64_t base, cudaStream_t s) {
    if (n <= 0) return;
    offsets_add_kernel<<<(unsigned)((n + kThreads - 1) / kThreads), kThreads, 0, s>>>(offsets, n, base);
    count_launches(1);
}

// Test hook (lbvh_test_hold_scan_tile): the tile that publishes nothing.
static std::atomic<int64_t> g_hold_scan_tile{-1};

void scan_set_hold_tile(int64_t tile) { g_hold_scan_tile.store(tile, std::memory_order_relaxed); }

void launch_exclusive_scan(const uint32_t *counts, int64_t nq, int64_t *offsets,
                           int64_t *tile_sums, Control *ctl, cudaStream_t s) {
    const int64_t tiles = nq > 0 ? scan_tile_count(nq) : 1;
    if (tiles <= kScanOnePass * (int64_t)device_sm_count()) {
        if (tiles > 1) cudaMemsetAsync(tile_sums, 0, (size_t)tiles * 8, s);
        scan_kernel<<<(unsigned)tiles, kScanThreads, 0, s>>>(counts, nq, reinterpret_cast<unsigned long long *>(tile_sums),
                                                             offsets, ctl,
                                                             g_hold_scan_tile.load(std::memory_order_relaxed));
        count_launches(1);
        return;
    }
    scan_reduce_kernel<<<(unsigned)tiles, kScanThreads, 0, s>>>(counts, nq, tile_sums);
    scan_tiles_kernel<<<1, kScanThreads, 0, s>>>(tile_sums, tiles, offsets, nq, &ctl->total);
    scan_apply_kernel<<<(unsigned)tiles, kScanThreads, 0, s>>>(counts, nq, tile_sums, offsets);
    count_launches(3);
}

}  // namespace lbvh
