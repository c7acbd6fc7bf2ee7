// construct.cu -- the single bottom-up pass of Algorithm 4 (Sec. 4): modified
// Apetrei merge that writes every internal node in Karras' ordering (Sec. 3.1)
// with its left child, its skip connection (Algorithm 2) and its box (Karras
// step 4, which Algorithm 4 leaves out; here the second thread up writes the
// union of its own box, held in registers, and its sibling's).
//
// One thread per leaf i:
//   1. delta*(i-1), delta*(i), delta*(i+1) from the sorted codes. delta is the
//      XOR reading of Sec. 3.2 with keys augmented by their sorted position:
//      64 + highest differing code bit, else the highest differing bit of the
//      positions; +inf (255) at -1 and n-1. Only comparisons are made and no
//      two compared gaps can share a highest bit, so this order is exact.
//   2. The leaf's skip (Algorithm 4's leaf lines) and box are written.
//   3. The nodes, without a climb wherever a warp can see both ends of a node's
//      range (merge_elements): a group of 128 consecutive leaves, in rounds of
//      32 elements to a warp, leaves about 7 open, which go to the group's
//      slots; merge_pending_kernel takes what 8 groups, then 5 of its own CTAs,
//      have left and merges it the same way (launch_merges says how far).
//   4. The rest climbs as Algorithm 4 does: a node's split p in its parent is
//      range_right (left child: delta_right < delta_left) or range_left - 1
//      (right child). The thread swaps its half of the parent's description
//      into store[p]. The first arrival reads "empty" and exits; the second
//      receives the other half, so it now knows the parent's full range [l, r]
//      and delta*(l-1), delta*(r), delta*(r+1). It computes the Karras index q
//      = r if delta*(r) < delta*(l-1) else l, the left child (L_p if l == p
//      else I_p: the children of split p are p and p+1), the skip (sentinel if
//      r == n-1, else L_{r+1} if delta*(r) < delta*(r+1), else I_{r+1}), and the
//      box, writes node q, and continues with i = q until q == 0 (I_0 is the
//      root in Karras' ordering).
//
// Differences from the listing, with the same result:
//   - store[p] carries, besides the range end, the delta* values the other
//     thread needs (packed into 64 bits), so no thread re-reads codes while
//     it climbs; only the leaf step reads codes, coalesced.
//   - an atomic exchange replaces compare-and-swap: exactly two threads
//     ever touch store[p], so the one that reads "empty" is the first. The
//     second writes "empty" back, leaving the scratch clean for the next build
//     (it is zeroed once, when allocated).
//   - release/acquire: the exchange is an acq_rel atomic, so a thread's node
//     is visible before its half of the parent is, and the second thread
//     reads the sibling's box (through L2, ld.global.cg) only after it has
//     seen that half.
//   - batches group their global sorted positions the same way (a group may
//     hold several trees; a split only ever joins leaves of one).
#include <atomic>

#include <cuda/atomic>

#include "lbvh_internal.cuh"
#include "morton.cuh"

namespace lbvh {

namespace {

constexpr uint32_t kInf = 255;  // above every finite delta* (<= 127)

__device__ __forceinline__ uint32_t delta_star(uint64_t a, uint64_t b, uint32_t pos) {
    const uint64_t x = a ^ b;
    if (x) return 127u - (uint32_t)__clzll((long long)x);  // 64 + highest differing bit
    return 31u - (uint32_t)__clz((int)(pos ^ (pos + 1u)));
}

// store word: bit 63 set = occupied.
//   left child's half (its range start l and delta*(l-1)):   l | d << 32
//   right child's half (range end r, delta*(r), delta*(r+1)): r | d << 32 | dn << 40
__device__ __forceinline__ unsigned long long pack(uint32_t end, uint32_t d, uint32_t dn) {
    return (1ull << 63) | ((unsigned long long)dn << 40) | ((unsigned long long)d << 32) | end;
}

template <int kKind>
__device__ __forceinline__ void load_node_box(const float4 *inodes, const float4 *leaves, int ni,
                                              int id, float3 &lo, float3 &hi) {
    if (id < ni) {
        const float4 a = __ldcg(inodes + 2 * (int64_t)id);
        const float4 b = __ldcg(inodes + 2 * (int64_t)id + 1);
        lo = make_float3(a.x, a.y, a.z);
        hi = make_float3(b.x, b.y, b.z);
    } else if (kKind == LBVH_PRIM_POINTS) {
        const float4 a = __ldcg(leaves + (id - ni));
        lo = make_float3(a.x, a.y, a.z);
        hi = lo;
    } else {
        const float4 a = __ldcg(leaves + 2 * (int64_t)(id - ni));
        const float4 b = __ldcg(leaves + 2 * (int64_t)(id - ni) + 1);
        lo = make_float3(a.x, a.y, a.z);
        hi = make_float3(b.x, b.y, b.z);
    }
}

// The exchange on store[p] publishes this thread's finished node (release)
// and, for the second thread, makes the sibling's node visible (acquire), as
// one acq_rel atomic. Measured with every exchange at device scope at 2^25
// points: 2.29 ms, against 2.96 ms for a relaxed exchange between two
// __threadfence() and 2.76 ms for a release-only exchange with an acquire
// fence taken by the second thread alone.
__device__ __forceinline__ unsigned long long publish_exchange(unsigned long long *slot, unsigned long long v) {
    cuda::atomic_ref<unsigned long long, cuda::thread_scope_device> a(*slot);
    return a.exchange(v, cuda::memory_order_acq_rel);
}

// Test hook (lbvh_test_construct_jitter): with kJitter, a thread waits a
// pseudo-random time of up to max_ns before each exchange (its delay drawn
// by splitmix64 from the seed and a salt naming the thread's place and
// level; %globaltimer, with an iteration cap as a backstop), so that the
// two children of a node arrive in other orders than the hardware's usual
// one. The kernels of every other build are instantiated without it.
struct Jitter {
    unsigned long long seed = 0;
    unsigned max_ns = 0;
};

template <bool kJitter>
__device__ __forceinline__ void jitter_wait(const Jitter &j, unsigned long long salt) {
    if constexpr (kJitter) {
        unsigned long long x = j.seed + (salt + 1ull) * 0x9e3779b97f4a7c15ull;
        x = (x ^ (x >> 30)) * 0xbf58476d1ce4e5b9ull;
        x = (x ^ (x >> 27)) * 0x94d049bb133111ebull;
        x ^= x >> 31;
        const unsigned long long d = x % ((unsigned long long)j.max_ns + 1ull);
        unsigned long long t0, t;
        asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t0));
        for (unsigned k = 0; k < (1u << 16); ++k) {
            asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
            if (t - t0 >= d) break;
        }
    }
}

// A thread's finished node while it climbs: leaf range [l, r], delta*(l-1),
// delta*(r), delta*(r+1), and its box.
struct Climb {
    uint32_t l, r, d_left, d_right, d_next;
    float3 lo, hi;
};

// The primitive's box (a point's box is the point).
template <int kKind>
__device__ __forceinline__ void gather_box(const float *__restrict__ prims, uint32_t p_id, float3 &lo, float3 &hi) {
    if (kKind == LBVH_PRIM_POINTS) {
        lo = make_float3(prims[3 * (int64_t)p_id], prims[3 * (int64_t)p_id + 1], prims[3 * (int64_t)p_id + 2]);
        hi = lo;
    } else {
        const float *b = prims + 6 * (int64_t)p_id;
        lo = make_float3(b[0], b[1], b[2]);
        hi = make_float3(b[3], b[4], b[5]);
    }
}

// Algorithm 4's leaf lines: leaf i of a tree of n leaves, own index p_own,
// box lo/hi, with delta*(i) and delta*(i+1).
template <int kKind>
__device__ __forceinline__ void leaf_write(int i, int n, uint32_t p_own, float3 lo, float3 hi, float4 *leaves,
                                           uint32_t dr, uint32_t drn) {
    // the leaf's skip is position i+1: one bit says I_{i+1} rather than L_{i+1}
    const uint32_t word = p_own | (i + 1 < n && dr >= drn ? kLeafSkipInternal : 0u);
    if (kKind == LBVH_PRIM_POINTS) {
        leaves[i] = make_float4(lo.x, lo.y, lo.z, __uint_as_float(word));
    } else {
        leaves[2 * (int64_t)i] = make_float4(lo.x, lo.y, lo.z, __uint_as_float(word));
        leaves[2 * (int64_t)i + 1] = make_float4(hi.x, hi.y, hi.z, 0.0f);
    }
}

// The parent's split p of c's node (range_right for a left child, range_left
// - 1 for a right child) and the half of the parent's description c gives.
__device__ __forceinline__ bool parent_split(const Climb &c, uint32_t &p, unsigned long long &mine) {
    const bool is_left = c.d_right < c.d_left;
    p = is_left ? c.r : c.l - 1;
    mine = is_left ? pack(c.l, c.d_left, 0) : pack(c.r, c.d_right, c.d_next);
    return is_left;
}

// The second thread up at split p takes the sibling's half: c becomes the
// parent's range; returns the sibling's node id (leaves from ni up).
__device__ __forceinline__ int take_half(Climb &c, bool is_left, uint32_t p, unsigned long long other,
                                         int ni) {
    if (is_left) {
        c.r = (uint32_t)other;
        c.d_right = (uint32_t)(other >> 32) & 0xffu;
        c.d_next = (uint32_t)(other >> 40) & 0xffu;
        return (p + 1 == c.r) ? ni + (int)p + 1 : (int)p + 1;
    }
    c.l = (uint32_t)other;
    c.d_left = (uint32_t)(other >> 32) & 0xffu;
    return (c.l == p) ? ni + (int)p : (int)p;
}

// The parent of split p: box = union with the sibling's, Karras index q = r
// if delta*(r) < delta*(l-1) else l, left child (L_p if l == p else I_p),
// skip (sentinel if r == n-1, else L_{r+1} if delta*(r) < delta*(r+1), else
// I_{r+1}). Writes node q and returns q.
__device__ __forceinline__ int write_parent(Climb &c, uint32_t p, int n, float3 slo, float3 shi,
                                            float4 *inodes) {
    const int ni = n - 1;
    c.lo = make_float3(min_ordered(c.lo.x, slo.x), min_ordered(c.lo.y, slo.y), min_ordered(c.lo.z, slo.z));
    c.hi = make_float3(max_ordered(c.hi.x, shi.x), max_ordered(c.hi.y, shi.y), max_ordered(c.hi.z, shi.z));
    const int q = c.d_right < c.d_left ? (int)c.r : (int)c.l;
    const int left_child = (c.l == p) ? ni + (int)p : (int)p;
    const int skip = (c.r == (uint32_t)(n - 1)) ? kSentinel
                                                : (c.d_right < c.d_next ? ni + (int)c.r + 1 : (int)c.r + 1);
    inodes[2 * (int64_t)q] = make_float4(c.lo.x, c.lo.y, c.lo.z, __int_as_float(left_child));
    inodes[2 * (int64_t)q + 1] = make_float4(c.hi.x, c.hi.y, c.hi.z, __int_as_float(skip));
    return q;
}

// Climb from c's node with device-scope exchanges on store[p] until this
// thread is the first up at a split, or has written the root I_0.
template <int kKind, bool kJitter = false>
__device__ __forceinline__ void climb_global(Climb c, int n, float4 *inodes, const float4 *leaves,
                                             unsigned long long *store, uint32_t *flags,
                                             const Jitter &jt = Jitter{}) {
    const int ni = n - 1;
    // The augmented keys have at most 64 + 32 bits, so no leaf is deeper than
    // 96 levels; the bound only guards against a corrupt input order.
    for (int level = 0; level < 128; ++level) {
        uint32_t p;
        unsigned long long mine;
        const bool is_left = parent_split(c, p, mine);
        if (p >= (uint32_t)ni) {
            atomicOr(flags, kFlagCorrupt);
            return;
        }
        jitter_wait<kJitter>(jt, (unsigned long long)p << 8 | (unsigned)level);
        const unsigned long long other = publish_exchange(store + p, mine);
        if (other == 0ull) return;  // first thread up
        store[p] = 0ull;            // second thread up: leave the slot empty again
        if ((uint32_t)other >= (uint32_t)n) {
            atomicOr(flags, kFlagCorrupt);
            return;
        }
        const int sibling = take_half(c, is_left, p, other, ni);
        float3 slo, shi;
        load_node_box<kKind>(inodes, leaves, ni, sibling, slo, shi);
        if (write_parent(c, p, n, slo, shi, inodes) == 0) return;  // the root
    }
    atomicOr(flags, kFlagCorrupt);
}

// Nodes inside a group of kGroup consecutive leaves, one group per CTA. A
// node of split p covers [l, r]: l - 1 and r are the nearest positions on
// either side whose delta* exceeds delta*(p). So a warp that holds 32
// consecutive elements (at first the leaves) has all it needs to write the
// nodes that both ends of which it can see, all at once: which lanes hold a
// larger gap comes from eight ballots, one to a bit of delta*, and the box of
// a range of lanes is the union of two entries of a table over runs of 2, 4,
// 8 and 16 lanes (min and max may count a lane twice). Splits whose range
// leaves the warp stay open; what lies between two open splits is one
// finished node (or leaf), an element of the next round. 128 leaves of
// uniform points leave 22 elements, then 7. What is left goes to the merges
// above the groups, or climbs with the device-scope exchanges of
// climb_global. The same nodes are written as by a climb from
// every leaf, each once.
//
// This is bound by instructions issued, not by memory. With a thread per
// leaf climbing through shared-memory words (block-scope exchanges, half the
// lanes gone after each level) this pass took 1226 instructions per warp of
// leaves and 1.57 ms at 2^25 points, 63-bit codes; now 757 and 1.14 (16,500
// points 31.7 -> 24.5 us, 1.0M 79.8 -> 64.4, 2^23 426 -> 311; a clustered
// mixture 41.9 -> 26.5, 92.1 -> 75.7, 438 -> 319, 2^25 1589 -> 1149). Groups of 128 leaves, 12 CTAs to
// an SM, against 256 with 6: 1.29 and 1.36 ms before the merges above them;
// 512: 1.48; 10 CTAs: 1.39. More CTAs take the L1's room for shared memory
// and the gathers miss: 14 CTAs 1.87.
constexpr int kGroup = 128;
constexpr int kWarps = kGroup / 32;
static_assert(kWarps == 4, "MergeSmem::count is one word");
constexpr int kGroupCtas = 12;  // CTAs of an SM
constexpr int kRuns = 4;  // runs of 2 .. 2^kRuns lanes in a warp's table

struct RunTable {
    float4 a[kRuns][32];  // lo.xyz, hi.x of the run that starts at a lane
    float2 b[kRuns][32];  // hi.yz
};

struct ElementList {
    uint32_t l[kGroup], r[kGroup], gaps[kGroup];
    float box[6][kGroup];
    int tree[kGroup];  // batches
};

// A merging CTA; the groups' CTAs also hold codes and gaps.
struct MergeSmem {
    union {
        uint64_t code[kGroup + 3];  // sorted codes a-1 .. a+kGroup+1
        RunTable table[kWarps];
        ElementList list;
    };
    alignas(4) uint8_t count[4];  // elements a warp leaves
    int failed;
};
struct GroupSmem : MergeSmem {
    uint8_t gap[kGroup + 4];  // delta* at a-1 .. a+kGroup (kInf between two trees)
    int instance[2];          // batches: of the first and the last leaf
};

// Elements left by a group: the CTA hands them, in order, to
// merge_pending_kernel through its own slots (16 bytes each: l, r, the three
// delta* values, the tree; the first one also carries how many there are, so
// only it has to be zero between builds). On uniform points a group of 128
// leaves has 7.3 of them on average, 1024 leaves 10.3, 7680 13.2, clustered
// ones 8.1, 12.3 and 15.7 (27 at most of 2,300). What a warp leaves always
// fits the slots, and 8 groups, or 5 CTAs of a merge, almost always fit a
// merge's 128 threads (with 256 the construct of 2^25 points took 1.23 ms, not
// 1.14; with 256 in the second merge alone 1.18). A longer list (chains of leaves
// with growing gaps) climbs in place and is marked kPendClimbed, and then the
// merge above climbs too. Where merges go to the end, its elements stay where
// they are instead: the last launch has a thread for every place of the lists
// before, and all that is left climbs there at once. (Where each merge waited for
// its own climbs, 64 clusters with points down to 1e-5 of their size, construct:
// 20,000 points 158 us, now 90; 24,000 boxes 168, 88; 7,000 points with 30 bits 93,
// 54. With all climbing from groups of 256: 98, 98, 51.)
constexpr int kPendSlots = 32;
constexpr int kPendCount = 24;  // first bit of the count
constexpr uint32_t kPendClimbed = 1u << 31;

struct Owner {  // a tree's leaves and memory
    int n;
    float4 *inodes;
    float4 *leaves;
    unsigned long long *store;
};

// A finished node or leaf: its leaves [l, r] in its tree, delta*(l-1) |
// delta*(r) << 8 | delta*(r+1) << 16, its box.
struct Element {
    uint32_t l, r, gaps;
    float3 lo, hi;
    int tree;
};

__device__ __forceinline__ float3 min3f(float3 a, float3 b) {
    return make_float3(min_ordered(a.x, b.x), min_ordered(a.y, b.y), min_ordered(a.z, b.z));
}
__device__ __forceinline__ float3 max3f(float3 a, float3 b) {
    return make_float3(max_ordered(a.x, b.x), max_ordered(a.y, b.y), max_ordered(a.z, b.z));
}
__device__ __forceinline__ float3 shfl_down3(float3 v, int by) {
    return make_float3(__shfl_down_sync(~0u, v.x, by), __shfl_down_sync(~0u, v.y, by), __shfl_down_sync(~0u, v.z, by));
}

// One warp over its first m lanes' elements (consecutive, m >= 1; all lanes
// call). Writes the nodes that are complete here; true where the lane's own
// split stays open: e is then the finished node or leaf that ends there.
// kPoint: e.lo == e.hi. owner(tree): the Owner.
template <bool kPoint, typename OwnerOf>
__device__ __forceinline__ bool merge_elements(RunTable &table, int m, Element &e, const OwnerOf &owner) {
    const int lane = threadIdx.x & 31;
    const bool have = lane < m;
    const uint32_t d = have ? (e.gaps >> 8) & 0xffu : 0u;
    // lanes with a larger gap, from the highest bit of delta* down
    uint32_t above = 0u, same = ~0u;
#pragma unroll
    for (int bit = 7; bit >= 0; --bit) {
        const uint32_t set = __ballot_sync(~0u, (d >> bit) & 1u);
        const uint32_t mine = (uint32_t)((int)(d << (31 - bit)) >> 31);  // all ones if the lane's bit is set
        above |= same & set & ~mine;
        same &= ~(set ^ mine);
    }
    const uint32_t before = (1u << lane) - 1u;
    const uint32_t lower = above & before, upper = above & ~before;
    const uint32_t outer = __shfl_sync(~0u, e.gaps, 0) & 0xffu;
    const bool complete = have && upper != 0u && (lower != 0u || outer > d);
    const uint32_t open = __ballot_sync(~0u, have && !complete);
    const uint32_t stops = complete ? lower : open & before;
    const int first = 32 - __clz((int)stops);
    const int last = complete ? __ffs((int)upper) - 1 : lane;
    const uint32_t p = e.r;
    const uint32_t l = __shfl_sync(~0u, e.l, first), r = __shfl_sync(~0u, e.r, last);
    const uint32_t left_gap = __shfl_sync(~0u, e.gaps, first) & 0xffu;
    const uint32_t right_gaps = __shfl_sync(~0u, e.gaps, last) & ~0xffu;
    // boxes of runs of 2, 4, 8, 16 lanes
    float3 lo = e.lo, hi = e.hi;
#pragma unroll
    for (int k = 0; k < kRuns; ++k) {
        const float3 nlo = shfl_down3(lo, 1 << k), nhi = k == 0 && kPoint ? nlo : shfl_down3(hi, 1 << k);
        lo = min3f(lo, nlo);
        hi = max3f(hi, nhi);
        table.a[k][lane] = make_float4(lo.x, lo.y, lo.z, hi.x);
        table.b[k][lane] = make_float2(hi.y, hi.z);
    }
    __syncwarp();
    const int len = last - first + 1;
    if (have && len > 1) {
        const int k = min(31 - __clz(len), kRuns) - 1;
        const int second = last + 1 - (2 << k);
        const float4 a0 = table.a[k][first], a1 = table.a[k][second];
        const float2 b0 = table.b[k][first], b1 = table.b[k][second];
        e.lo = min3f(make_float3(a0.x, a0.y, a0.z), make_float3(a1.x, a1.y, a1.z));
        e.hi = max3f(make_float3(a0.w, b0.x, b0.y), make_float3(a1.w, b1.x, b1.y));
    }
    e.l = l;
    e.r = r;
    e.gaps = left_gap | right_gaps;
    if (complete) {
        const Owner o = owner(e.tree);
        const int ni = o.n - 1;
        const uint32_t dr = (right_gaps >> 8) & 0xffu;
        const int q = (int)(dr < left_gap ? r : l);
        const int left_child = (int)(l == p ? ni + p : p);
        const int skip = dr == kInf ? kSentinel : (int)(dr < right_gaps >> 16 ? ni + r + 1 : r + 1);
        o.inodes[2 * (int64_t)q] = make_float4(e.lo.x, e.lo.y, e.lo.z, __int_as_float(left_child));
        o.inodes[2 * (int64_t)q + 1] = make_float4(e.hi.x, e.hi.y, e.hi.z, __int_as_float(skip));
    }
    return have && !complete;
}

// A CTA's elements, consecutive, one per thread (the first `count`): merges
// them in rounds; what is left goes to the CTA's slots (pend), or, if it is too
// much for them, to lists at `back` (room for kGroup elements), or climbs.
// Every thread of the CTA calls this; the tables' memory is free.
template <int kKind, bool kPoints, bool kJitter, bool kTrees, typename OwnerOf>
__device__ __forceinline__ void merge_group(MergeSmem &sm, int count, Element e, const OwnerOf &owner,
                                            uint32_t *flags, uint4 *pend, const Jitter &jt, uint4 *back = nullptr) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    bool keep = false;
    uint32_t kept = 0u;
    int at = 0, left = 0;  // the element's place among those left, and their number
    for (int round = 0;; ++round) {
        const int m = min(count - 32 * warp, 32);
        keep = false;
        if (m > 0) {
            keep = kPoints && round == 0 ? merge_elements<true>(sm.table[warp], m, e, owner)
                                         : merge_elements<false>(sm.table[warp], m, e, owner);
            // a whole tree is done (its root is written, or it is one leaf)
            keep = keep && (e.gaps & 0xffffu) != (kInf | kInf << 8);
        }
        kept = __ballot_sync(~0u, keep);
        at = __popc(kept & ((1u << lane) - 1u));
        left = __popc(kept);
        if (count <= 32) break;  // all of them the first warp's
        if (lane == 0) sm.count[warp] = (uint8_t)left;
        __syncthreads();  // also: every warp is through with its table
        const uint32_t counts = *reinterpret_cast<const uint32_t *>(sm.count);  // a byte per warp
        at += (int)__dp4a(counts & ((1u << (8 * warp)) - 1u), 0x01010101u, 0u);
        left = (int)__dp4a(counts, 0x01010101u, 0u);
        if (left == count) break;  // no warp could merge anything
        count = left;
        if (keep) {
            sm.list.l[at] = e.l;
            sm.list.r[at] = e.r;
            sm.list.gaps[at] = e.gaps;
            sm.list.box[0][at] = e.lo.x;
            sm.list.box[1][at] = e.lo.y;
            sm.list.box[2][at] = e.lo.z;
            sm.list.box[3][at] = e.hi.x;
            sm.list.box[4][at] = e.hi.y;
            sm.list.box[5][at] = e.hi.z;
            if (kTrees) sm.list.tree[at] = e.tree;
        }
        __syncthreads();
        if ((int)threadIdx.x < count) {
            const int k = threadIdx.x;
            e.l = sm.list.l[k];
            e.r = sm.list.r[k];
            e.gaps = sm.list.gaps[k];
            e.lo = make_float3(sm.list.box[0][k], sm.list.box[1][k], sm.list.box[2][k]);
            e.hi = make_float3(sm.list.box[3][k], sm.list.box[4][k], sm.list.box[5][k]);
            if (kTrees) e.tree = sm.list.tree[k];
        }
        __syncthreads();  // the tables take the list's place
    }
    const bool one_warp = count <= 32;  // what is left, and the last round's nodes: the first warp's
    if (pend && (one_warp ? __popc(kept) : left) <= kPendSlots) {
        if (keep)
            pend[at] = make_uint4(e.l, e.r, e.gaps | (at == 0 ? (uint32_t)left << kPendCount : 0u), (uint32_t)e.tree);
        return;
    }
    if (pend && threadIdx.x == 0) pend[0] = make_uint4(0u, 0u, kPendClimbed, 0u);
    if (back) {  // (over kPendSlots elements: the barriers above come after the lists there were cleared)
        const uint32_t listed = at % kPendSlots == 0 ? (uint32_t)min(left - at, kPendSlots) << kPendCount : 0u;
        if (keep) back[at] = make_uint4(e.l, e.r, e.gaps | listed, (uint32_t)e.tree);
        return;
    }
    // The nodes of this CTA, whichever thread wrote them, are visible to
    // whoever sees this thread's exchange: the barrier orders them before its
    // release.
    if (one_warp) __syncwarp();
    else __syncthreads();
    if (!keep) return;
    const Owner o = owner(e.tree);
    climb_global<kKind, kJitter>(Climb{e.l, e.r, e.gaps & 0xffu, (e.gaps >> 8) & 0xffu, (e.gaps >> 16) & 0xffu, e.lo, e.hi},
                                 o.n, o.inodes, o.leaves, o.store, flags, jt);
}

// The build's error flags, read once per CTA (they go to sm.failed before the
// CTA's first barrier): if an earlier stage failed, the whole CTA returns and
// leaves `store` untouched.
__device__ __forceinline__ void group_start(MergeSmem &sm, const uint32_t *flags) {
    if (threadIdx.x == 0) sm.failed = (__ldcg(flags) & (kFlagTimeout | kFlagCorrupt)) != 0;
}

struct OneTree {
    Owner o;
    __device__ __forceinline__ Owner operator()(int) const { return o; }
};

// The trees of a batch: global sorted position g belongs to the instance b
// with off[b] <= g < off[b+1]; its tree's records start at node_start[b]
// (float4 units) and its store words at store_start[b].
struct ManyTrees {
    const int64_t *off, *node_start, *store_start;
    float4 *nodes;
    unsigned long long *store;
    __device__ __forceinline__ Owner operator()(int b) const {
        const int n = (int)(__ldg(off + b + 1) - __ldg(off + b));
        float4 *inodes = nodes + __ldg(node_start + b);
        return Owner{n, inodes, inodes + 2 * (int64_t)(n - 1), store + __ldg(store_start + b)};
    }
};

// What kMergeGroups groups left (then kMergeCtas CTAs of a merge) is merged the
// same way, the nodes read back for their boxes. With a thread per element
// climbing from there the construct of 2^25 points took 1.29 ms, so 1.13; 512
// batched trees of 36,000 points that climbed inside the groups' kernel 1.13
// ms, so 0.60.
constexpr int kMergeGroups = 8;
constexpr int kMergeCtas = 5;

// The lists an earlier merge read.
struct Lists {
    uint4 *pend;
    int64_t count;
    __host__ __device__ int64_t ctas() const { return (count * kPendSlots + kGroup - 1) / kGroup; }
};
constexpr int kEarlier = 2;
struct EarlierMerges {
    Lists level[kEarlier];
};

// merging: the CTAs that merge; those beyond (the last launch of several) climb
// from what the merges before have left. defer: leave what does not fit.
template <int kKind, int kFrom, bool kJitter, bool kTrees, typename OwnerOf>
__global__ void __launch_bounds__(kGroup)
    merge_pending_kernel(uint4 *pend, int64_t lists, OwnerOf owner, uint32_t *flags, uint4 *out, Jitter jt, bool defer,
                         unsigned merging, EarlierMerges earlier) {
    __shared__ MergeSmem sm;
    __shared__ uint32_t s_lists[kFrom];
    group_start(sm, flags);
    const int t = threadIdx.x;
    if (out) out += (int64_t)blockIdx.x * kPendSlots;
    pend += (int64_t)blockIdx.x * kFrom * kPendSlots;
    const bool list = t < kFrom && (int64_t)blockIdx.x * kFrom + t < lists;
    if (t < kFrom) s_lists[t] = list ? pend[t * kPendSlots].z : 0u;
    __syncthreads();
    int count = 0;
    bool missing = false;
#pragma unroll
    for (int k = 0; k < kFrom; ++k) {
        count += (int)(s_lists[k] >> kPendCount) & 127;
        missing = missing || (s_lists[k] & kPendClimbed) != 0u;
    }
    // the j-th element, counted through the lists
    const auto place = [&](int j) {
        int before = 0, at = j;
#pragma unroll
        for (int k = 0; k < kFrom; ++k) {
            if (j >= before) at = k * kPendSlots + j - before;
            before += (int)(s_lists[k] >> kPendCount) & 127;
        }
        return at;
    };
    const auto element = [&](const uint4 &w) {
        Element e{w.x, w.y, w.z & 0xffffffu, make_float3(0.f, 0.f, 0.f), make_float3(0.f, 0.f, 0.f), (int)w.w};
        const Owner o = owner(e.tree);
        // the node of range [l, r]: leaf l, or internal node r or l (its Karras index)
        const uint32_t dl = e.gaps & 0xffu, dr = (e.gaps >> 8) & 0xffu;
        const int id = (int)(e.l == e.r ? (uint32_t)(o.n - 1) + e.l : (dr < dl ? e.r : e.l));
        load_node_box<kKind>(o.inodes, o.leaves, o.n - 1, id, e.lo, e.hi);
        return e;
    };
    const auto climb = [&](const Element &e) {
        const Owner o = owner(e.tree);
        climb_global<kKind, kJitter>(Climb{e.l, e.r, e.gaps & 0xffu, (e.gaps >> 8) & 0xffu, (e.gaps >> 16) & 0xffu, e.lo, e.hi},
                                     o.n, o.inodes, o.leaves, o.store, flags, jt);
    };
    if (blockIdx.x >= merging) {  // a thread for every place of four of the lists before
        int64_t b = blockIdx.x - merging;
        int lv = 0;
        while (lv + 1 < kEarlier && b >= earlier.level[lv].ctas()) b -= earlier.level[lv++].ctas();
        const Lists left = earlier.level[lv];
        uint4 *at = left.pend + b * kGroup;
        const bool there = b * kGroup / kPendSlots + t / kPendSlots < left.count;
        const uint32_t listed = there ? (at[t / kPendSlots * kPendSlots].z >> kPendCount) & 127u : 0u;
        if (t % kPendSlots < (int)listed && !sm.failed) climb(element(at[t]));
        __syncthreads();
        if (there && t % kPendSlots == 0) at[t].z = 0u;
        return;
    }
    if (defer && !sm.failed && (missing || count > kGroup)) {
        if (t == 0) out[0] = make_uint4(0u, 0u, kPendClimbed, 0u);
        return;
    }
    if (sm.failed || missing || count > kGroup) {
        // failed: only the counts are cleared; else (some elements missing, or too many) those that are here climb
        if (out && t == 0 && !sm.failed) out[0] = make_uint4(0u, 0u, kPendClimbed, 0u);
        for (int k = t; k < count && !sm.failed; k += kGroup) climb(element(pend[place(k)]));
        __syncthreads();
        if (list) pend[t * kPendSlots].z = 0u;
        return;
    }
    Element e{};
    if (t < count) e = element(pend[place(t)]);
    __syncthreads();
    if (list) pend[t * kPendSlots].z = 0u;
    merge_group<kKind, false, kJitter, kTrees>(sm, count, e, owner, flags, out, jt, defer ? pend : nullptr);
}

// delta* at the CTA's positions, from sm.code. Thread t holds leaf i of a
// tree of n leaves (i >= n: no leaf). Codes out of order latch kFlagCorrupt:
// the input is not sorted.
__device__ __forceinline__ void group_gaps(GroupSmem &sm, int i, int n, uint32_t *flags) {
    const int t = threadIdx.x;
    uint32_t dr = kInf;
    if (i + 1 < n) {
        const uint64_t c0 = sm.code[t + 1], c1 = sm.code[t + 2];
        if (c0 > c1) atomicOr(flags, kFlagCorrupt);
        dr = delta_star(c0, c1, (uint32_t)i);
    }
    sm.gap[t + 1] = (uint8_t)dr;
    if (t == 0) sm.gap[0] = (uint8_t)(i > 0 && i < n ? delta_star(sm.code[0], sm.code[1], (uint32_t)(i - 1)) : kInf);
    if (t == kGroup - 1)
        sm.gap[kGroup + 1] =
            (uint8_t)(i + 2 < n ? delta_star(sm.code[t + 2], sm.code[t + 3], (uint32_t)(i + 1)) : kInf);
}

// Leaf i's element: its gaps, in place in sm.gap.
__device__ __forceinline__ uint32_t leaf_gaps(const GroupSmem &sm) {
    const int t = threadIdx.x;
    return sm.gap[t] | (uint32_t)sm.gap[t + 1] << 8 | (uint32_t)sm.gap[t + 2] << 16;
}

// Algorithm 4 from sorted codes and a permutation (lbvh_build_from_sorted,
// refit, the no-allocation entry point).
template <int kKind, bool kJitter>
__global__ void __launch_bounds__(kGroup, kGroupCtas)
    construct_block_kernel(const uint64_t *__restrict__ codes, const uint32_t *__restrict__ perm,
                           const float *__restrict__ prims, int n, float4 *inodes, float4 *leaves,
                           unsigned long long *store, uint32_t *flags, uint4 *pend, Jitter jt) {
    __shared__ GroupSmem sm;
    group_start(sm, flags);
    const int t = threadIdx.x;
    const int64_t a = (int64_t)blockIdx.x * kGroup;
    const int i = (int)a + t;
    const bool mine = i < n;
    const uint32_t p_id = mine ? perm[i] : 0u;
    const bool ok = mine && p_id < (uint32_t)n;
    Element e{(uint32_t)i, (uint32_t)i, 0u, make_float3(0.f, 0.f, 0.f), make_float3(0.f, 0.f, 0.f), 0};
    if (ok) gather_box<kKind>(prims, p_id, e.lo, e.hi);
    if (mine) sm.code[t + 1] = codes[i];
    if (t < 3) {
        const int64_t h = t == 0 ? a - 1 : a + kGroup + t - 1;
        if (h >= 0 && h < n) sm.code[t == 0 ? 0 : kGroup + t] = codes[h];
    }
    __syncthreads();
    if (sm.failed) return;
    if (mine && !ok) atomicOr(flags, kFlagCorrupt);  // not a permutation: the sort failed
    group_gaps(sm, i, n, flags);
    __syncthreads();
    e.gaps = leaf_gaps(sm);
    if (ok) leaf_write<kKind>(i, n, p_id, e.lo, e.hi, leaves, (e.gaps >> 8) & 0xffu, e.gaps >> 16);
    merge_group<kKind, kKind == LBVH_PRIM_POINTS, kJitter, false>(
        sm, (int)min((int64_t)kGroup, n - a), e, OneTree{Owner{n, inodes, leaves, store}}, flags,
        pend ? pend + (int64_t)blockIdx.x * kPendSlots : nullptr, jt);
}

// Algorithm 4 after a sort that kept only the permutation. Each thread
// gathers its leaf's primitive and derives its Morton code again with the
// encoder's function (the same bits); the codes of the CTA's leaves and of
// three neighbours (positions a-1, a+kGroup, a+kGroup+1, gathered by threads
// 0-2) meet in shared memory for the delta* values. The sorted codes are
// written to codes_out (the tree keeps them for export and refit).
template <int kKind, bool kJitter>
__global__ void __launch_bounds__(kGroup, kGroupCtas)
    construct_encode_kernel(const uint32_t *__restrict__ perm, const float *__restrict__ prims,
                            const float *__restrict__ bounds, int b, int n, uint64_t *__restrict__ codes_out,
                            float4 *inodes, float4 *leaves, unsigned long long *store, uint32_t *flags,
                            uint4 *pend, Jitter jt) {
    __shared__ GroupSmem sm;
    group_start(sm, flags);
    const int t = threadIdx.x;
    const int64_t a = (int64_t)blockIdx.x * kGroup;
    const int i = (int)a + t;
    const Grid3 g = make_grid(bounds, b);
    const bool mine = i < n;
    const uint32_t p_id = mine ? __ldcs(perm + i) : 0u;
    const bool ok = mine && p_id < (uint32_t)n;
    Element e{(uint32_t)i, (uint32_t)i, 0u, make_float3(0.f, 0.f, 0.f), make_float3(0.f, 0.f, 0.f), 0};
    if (ok) gather_box<kKind>(prims, p_id, e.lo, e.hi);
    // the three neighbours outside the CTA's range
    int64_t hpos = -1;
    float3 hlo = e.lo, hhi = e.hi;
    if (t < 3) {
        hpos = t == 0 ? a - 1 : a + kGroup + t - 1;
        if (hpos >= 0 && hpos < n) {
            const uint32_t hp = perm[hpos];
            if (hp < (uint32_t)n) gather_box<kKind>(prims, hp, hlo, hhi);
            else hpos = -1;
        } else {
            hpos = -1;
        }
    }
    uint64_t code = 0;
    if (mine) {
        code = morton(__fmul_rn(__fadd_rn(e.lo.x, e.hi.x), 0.5f), __fmul_rn(__fadd_rn(e.lo.y, e.hi.y), 0.5f),
                      __fmul_rn(__fadd_rn(e.lo.z, e.hi.z), 0.5f), g);
        sm.code[t + 1] = code;
    }
    if (hpos >= 0)
        sm.code[t == 0 ? 0 : kGroup + t] =
            morton(__fmul_rn(__fadd_rn(hlo.x, hhi.x), 0.5f), __fmul_rn(__fadd_rn(hlo.y, hhi.y), 0.5f),
                   __fmul_rn(__fadd_rn(hlo.z, hhi.z), 0.5f), g);
    __syncthreads();
    if (sm.failed) return;
    if (ok) codes_out[i] = code;
    if (mine && !ok) atomicOr(flags, kFlagCorrupt);  // not a permutation: the sort failed
    group_gaps(sm, i, n, flags);
    __syncthreads();
    e.gaps = leaf_gaps(sm);
    if (ok) leaf_write<kKind>(i, n, p_id, e.lo, e.hi, leaves, (e.gaps >> 8) & 0xffu, e.gaps >> 16);
    merge_group<kKind, kKind == LBVH_PRIM_POINTS, kJitter, false>(
        sm, (int)min((int64_t)kGroup, n - a), e, OneTree{Owner{n, inodes, leaves, store}}, flags,
        pend ? pend + (int64_t)blockIdx.x * kPendSlots : nullptr, jt);
}

// Many trees at once, grouped by global sorted position.
template <int kKind>
__global__ void __launch_bounds__(kGroup, kGroupCtas)
    batch_construct_block_kernel(const uint64_t *__restrict__ codes, const uint32_t *__restrict__ perm,
                                 const float *__restrict__ prims, const int64_t *__restrict__ off,
                                 const int64_t *__restrict__ node_start, const int64_t *__restrict__ store_start,
                                 int count, int64_t total, float4 *nodes, unsigned long long *store,
                                 uint32_t *flags, uint4 *pend) {
    __shared__ GroupSmem sm;
    group_start(sm, flags);
    const int t = threadIdx.x;
    const int64_t a = (int64_t)blockIdx.x * kGroup, g = a + t;
    const bool mine = g < total;
    if (mine) sm.code[t + 1] = codes[g];
    if (t < 3) {
        const int64_t h = t == 0 ? a - 1 : a + kGroup + t - 1;
        if (h >= 0 && h < total) sm.code[t == 0 ? 0 : kGroup + t] = codes[h];
    }
    const uint32_t p_id = mine ? perm[g] : 0u;
    // the instance: most groups lie in one, which the two ends show
    if (t == 0) sm.instance[0] = instance_of(off, count, a);
    if (t == 32) sm.instance[1] = instance_of(off, count, min(a + kGroup, total) - 1);
    __syncthreads();
    if (sm.failed) return;
    int b = sm.instance[0];
    if (mine && b < sm.instance[1]) b += instance_of(off + b, sm.instance[1] - b + 1, g);
    const ManyTrees owner{off, node_start, store_start, nodes, store};
    const Owner o = owner(b);
    const int64_t base = __ldg(off + b);
    const int i = mine ? (int)(g - base) : o.n;
    const uint32_t p_own = p_id - (uint32_t)base;
    const bool ok = mine && p_own < (uint32_t)o.n;
    Element e{(uint32_t)i, (uint32_t)i, 0u, make_float3(0.f, 0.f, 0.f), make_float3(0.f, 0.f, 0.f), b};
    if (ok) gather_box<kKind>(prims, p_id, e.lo, e.hi);
    if (mine && !ok) atomicOr(flags, kFlagCorrupt);  // not a permutation of this tree: the sort failed
    group_gaps(sm, i, o.n, flags);
    __syncthreads();
    e.gaps = leaf_gaps(sm);
    if (ok) leaf_write<kKind>(i, o.n, p_own, e.lo, e.hi, o.leaves, (e.gaps >> 8) & 0xffu, e.gaps >> 16);
    merge_group<kKind, kKind == LBVH_PRIM_POINTS, false, true>(sm, (int)min((int64_t)kGroup, total - a), e, owner, flags,
                                                               pend + (int64_t)blockIdx.x * kPendSlots, Jitter{});
}

// How far the merges go before the rest climbs. A merge is a launch of about
// 6 us that its CTAs' own latency sets, a climb 1-2 us per level of the tree;
// where a list is too long, what waits for it climbs all the same. So only
// small builds merge to the end: 16,500 points, clustered or not, 24.5 us
// against 29.6 to 36.8 (100,000 32.7 against 35 to 43, but the last launch's
// threads for the lists before grow with the build).
// Merging again while there are over 4096 CTAs (2^25 points): 1.14 ms, never
// 1.27, to the end (mixture) 1.48.
constexpr int64_t kMergeToEnd = 24;
constexpr int64_t kMergeAgain = 4096;

int64_t merge_ctas(int64_t lists, bool groups) {
    const int64_t each = groups ? kMergeGroups : kMergeCtas;
    return (lists + each - 1) / each;
}

template <bool kTrees, typename OwnerOf>
void launch_merges(int64_t groups, int kind, const OwnerOf &owner, uint32_t *flags, void *pend, const Jitter &jt,
                   cudaStream_t s) {
    if (!pend || groups < 2) return;  // one group leaves nothing
    uint4 *in = static_cast<uint4 *>(pend);
    int64_t from = groups;
    const bool to_end = merge_ctas(groups, true) <= kMergeToEnd && jt.max_ns == 0;
    int64_t enough = to_end ? 1 : kMergeAgain;
    EarlierMerges earlier{};
    int merges = 0;
    if (jt.max_ns) enough = groups;  // the hook is for climbs: what the first merge leaves climbs
    static_assert(kMergeToEnd <= kMergeCtas * kMergeCtas, "at most kEarlier merges before the last");
    const bool pts = kind == LBVH_PRIM_POINTS;
    for (bool first = true;; first = false) {
        const int64_t ctas = merge_ctas(from, first);
        uint4 *out = ctas > enough ? in + from * kPendSlots : nullptr;
        const auto pick = [&](auto a, auto b, auto c, auto d) { return first ? (pts ? a : b) : (pts ? c : d); };
        auto k = pick(merge_pending_kernel<LBVH_PRIM_POINTS, kMergeGroups, false, kTrees, OwnerOf>,
                      merge_pending_kernel<LBVH_PRIM_BOXES, kMergeGroups, false, kTrees, OwnerOf>,
                      merge_pending_kernel<LBVH_PRIM_POINTS, kMergeCtas, false, kTrees, OwnerOf>,
                      merge_pending_kernel<LBVH_PRIM_BOXES, kMergeCtas, false, kTrees, OwnerOf>);
        if constexpr (!kTrees) {
            if (jt.max_ns)
                k = pick(merge_pending_kernel<LBVH_PRIM_POINTS, kMergeGroups, true, kTrees, OwnerOf>,
                         merge_pending_kernel<LBVH_PRIM_BOXES, kMergeGroups, true, kTrees, OwnerOf>,
                         merge_pending_kernel<LBVH_PRIM_POINTS, kMergeCtas, true, kTrees, OwnerOf>,
                         merge_pending_kernel<LBVH_PRIM_BOXES, kMergeCtas, true, kTrees, OwnerOf>);
        }
        int64_t more = 0;  // what the merges to the end leave climbs in the last one
        if (!out)
            for (const Lists &l : earlier.level) more += l.ctas();
        k<<<(unsigned)(ctas + more), kGroup, 0, s>>>(in, from, owner, flags, out, jt, to_end && out, (unsigned)ctas, earlier);
        count_launches(1);
        if (!out) return;
        if (to_end) earlier.level[merges++] = Lists{in, from};
        in = out;
        from = ctas;
    }
}

}  // namespace

size_t construct_pend_bytes(int64_t n) {
    int64_t from = (n + kGroup - 1) / kGroup, slots = from * kPendSlots;
    for (bool first = true; from > 1; first = false) {
        from = merge_ctas(from, first);
        slots += from * kPendSlots;
    }
    return (size_t)slots * sizeof(uint4);
}

void launch_batch_construct(const uint64_t *sorted_codes, const uint32_t *perm, const float *prims,
                            const BatchTables &bt, int kind, float4 *nodes, unsigned long long *store,
                            uint32_t *flags, void *pend, cudaStream_t s) {
    if (bt.total_prims <= 0) return;
    const unsigned blocks = (unsigned)((bt.total_prims + kGroup - 1) / kGroup);
    auto k = kind == LBVH_PRIM_POINTS ? batch_construct_block_kernel<LBVH_PRIM_POINTS>
                                      : batch_construct_block_kernel<LBVH_PRIM_BOXES>;
    k<<<blocks, kGroup, 0, s>>>(sorted_codes, perm, prims, bt.prim_off, bt.node_start, bt.store_start, bt.count,
                                bt.total_prims, nodes, store, flags, static_cast<uint4 *>(pend));
    count_launches(1);
    launch_merges<true>(blocks, kind, ManyTrees{bt.prim_off, bt.node_start, bt.store_start, nodes, store}, flags, pend,
                        Jitter{}, s);
}

namespace {

// lbvh_test_construct_jitter's setting (max_ns 0: off)
std::atomic<unsigned long long> g_jitter_seed{0};
std::atomic<unsigned> g_jitter_ns{0};

Jitter jitter_setting() {
    Jitter j;
    j.seed = g_jitter_seed.load(std::memory_order_relaxed);
    j.max_ns = g_jitter_ns.load(std::memory_order_relaxed);
    return j;
}

}  // namespace

void launch_construct(const uint64_t *sorted_codes, const uint32_t *perm, const float *prims,
                      int64_t n, int kind, float4 *inodes, float4 *leaves,
                      unsigned long long *store, uint32_t *flags, void *pend, cudaStream_t s) {
    if (n <= 0) return;
    const unsigned blocks = (unsigned)((n + kGroup - 1) / kGroup);
    const Jitter jt = jitter_setting();
    const bool pts = kind == LBVH_PRIM_POINTS;
    auto k = jt.max_ns ? (pts ? construct_block_kernel<LBVH_PRIM_POINTS, true>
                              : construct_block_kernel<LBVH_PRIM_BOXES, true>)
                       : (pts ? construct_block_kernel<LBVH_PRIM_POINTS, false>
                              : construct_block_kernel<LBVH_PRIM_BOXES, false>);
    k<<<blocks, kGroup, 0, s>>>(sorted_codes, perm, prims, (int)n, inodes, leaves, store, flags,
                                static_cast<uint4 *>(pend), jt);
    count_launches(1);
    launch_merges<false>(blocks, kind, OneTree{Owner{(int)n, inodes, leaves, store}}, flags, pend, jt, s);
}

void launch_construct_encode(const uint32_t *perm, const float *prims, const float *bounds, int bits, int64_t n,
                             int kind, uint64_t *codes_out, float4 *inodes, float4 *leaves,
                             unsigned long long *store, uint32_t *flags, void *pend, cudaStream_t s) {
    if (n <= 0) return;
    const unsigned blocks = (unsigned)((n + kGroup - 1) / kGroup);
    const Jitter jt = jitter_setting();
    const bool pts = kind == LBVH_PRIM_POINTS;
    auto k = jt.max_ns ? (pts ? construct_encode_kernel<LBVH_PRIM_POINTS, true>
                              : construct_encode_kernel<LBVH_PRIM_BOXES, true>)
                       : (pts ? construct_encode_kernel<LBVH_PRIM_POINTS, false>
                              : construct_encode_kernel<LBVH_PRIM_BOXES, false>);
    k<<<blocks, kGroup, 0, s>>>(perm, prims, bounds, bits / 3, (int)n, codes_out, inodes, leaves, store, flags,
                                static_cast<uint4 *>(pend), jt);
    count_launches(1);
    launch_merges<false>(blocks, kind, OneTree{Owner{(int)n, inodes, leaves, store}}, flags, pend, jt, s);
}

}  // namespace lbvh

// ---------------------------------------------------------------- no-allocation variant
//
// lbvh_construct_static runs the same construct kernel as the tree builds,
// with Algorithm 4's `store` words in a file-scope device array instead of
// memory the library allocates. The array is as large as the biggest tree the
// entry point accepts, and every GPU that loads this library holds it until
// the process exits.
namespace {

constexpr int64_t kStaticMaxPrims = (int64_t(1) << 20) + 1;  // store words: n - 1 <= 2^20 (8 MiB)

__device__ __align__(256) unsigned long long g_static_store[kStaticMaxPrims - 1];
__device__ __align__(256) uint32_t g_static_flags[64];

// Device addresses of the two arrays for the current device. Host code must
// not use the symbols themselves (in host code they name host-side stand-ins).
// The lookup is repeated on every call: it is cheap, and an address kept from
// an earlier call would go stale if the caller reset the device (the module,
// and with it the arrays, is loaded again into the new context).
struct StaticScratch {
    unsigned long long *store = nullptr;
    uint32_t *flags = nullptr;
};

lbvh_status static_scratch(StaticScratch *out) {
    void *store = nullptr, *flags = nullptr;
    if (cudaGetSymbolAddress(&store, g_static_store) != cudaSuccess) return LBVH_ERR_CUDA;
    if (cudaGetSymbolAddress(&flags, g_static_flags) != cudaSuccess) return LBVH_ERR_CUDA;
    out->store = static_cast<unsigned long long *>(store);
    out->flags = static_cast<uint32_t *>(flags);
    return LBVH_OK;
}

}  // namespace

extern "C" lbvh_status lbvh_test_construct_jitter(unsigned long long seed, unsigned max_ns) {
    if (max_ns > 1000000u) return LBVH_ERR_INVALID;
    lbvh::g_jitter_seed.store(seed, std::memory_order_relaxed);
    lbvh::g_jitter_ns.store(max_ns, std::memory_order_relaxed);
    return LBVH_OK;
}

extern "C" lbvh_status lbvh_construct_static(const uint64_t *d_sorted_codes, const uint32_t *d_perm,
                                             const float *d_prims, int64_t n, int kind, float *d_inodes,
                                             float *d_leaves, uint32_t *d_flags, lbvh_stream_t stream) {
    if (n < 1 || n > kStaticMaxPrims) return LBVH_ERR_INVALID;
    if (kind != LBVH_PRIM_POINTS && kind != LBVH_PRIM_BOXES) return LBVH_ERR_INVALID;
    if (!d_sorted_codes || !d_perm || !d_prims || !d_leaves || (n > 1 && !d_inodes)) return LBVH_ERR_INVALID;
    (void)cudaGetLastError();  // an earlier, unrelated error must not be charged to this call
    StaticScratch scratch;
    const lbvh_status st = static_scratch(&scratch);
    if (st != LBVH_OK) return st;
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    // every call shares the array: the store words must start empty (zero)
    if (n > 1 && cudaMemsetAsync(scratch.store, 0, (size_t)(n - 1) * sizeof(unsigned long long), s) != cudaSuccess)
        return LBVH_ERR_CUDA;
    uint32_t *flags = d_flags;
    if (!flags) {
        flags = scratch.flags;
        if (cudaMemsetAsync(flags, 0, sizeof(uint32_t), s) != cudaSuccess) return LBVH_ERR_CUDA;
    }
    lbvh::launch_construct(d_sorted_codes, d_perm, d_prims, n, kind, reinterpret_cast<float4 *>(d_inodes),
                           reinterpret_cast<float4 *>(d_leaves), scratch.store, flags, nullptr, s);
    return cudaGetLastError() == cudaSuccess ? LBVH_OK : LBVH_ERR_CUDA;
}

