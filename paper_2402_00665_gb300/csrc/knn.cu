// knn.cu -- k nearest neighbours: the distance range search of Sec. 1 asked
// for its k closest answers. One thread per query with a heap and Algorithm 1
// (heap_walk), or packets of query points through the leaf blocks.
#include <algorithm>
#include <type_traits>

#include "lbvh_internal.cuh"
#include "morton.cuh"
#include "packet.cuh"
#include "walk.cuh"

namespace lbvh {

namespace {

// Max-heap of (squared distance bits << 32 | primitive index) keys in the
// thread's local memory: keys order like (distance, index), distances being
// non-negative floats.
template <int kCap>
struct KnnHeap {
    uint64_t h[kCap];
    int cnt;

    __device__ __forceinline__ void push(uint64_t key) {
        int i = cnt++;
        while (i > 0) {
            const int p = (i - 1) >> 1;
            if (h[p] >= key) break;
            h[i] = h[p];
            i = p;
        }
        h[i] = key;
    }
    // the largest key leaves and `key` (smaller than it) enters
    __device__ __forceinline__ void sift_from_top(uint64_t key, int size) {
        int i = 0;
        while (true) {
            const int l = 2 * i + 1;
            if (l >= size) break;
            const int r = l + 1;
            const int c = (r < size && h[r] > h[l]) ? r : l;
            if (h[c] <= key) break;
            h[i] = h[c];
            i = c;
        }
        h[i] = key;
    }
    // heap sort: ascending keys in h[0..cnt)
    __device__ __forceinline__ void sort() {
        for (int e = cnt - 1; e > 0; --e) {
            const uint64_t top = h[0];
            sift_from_top(h[e], e);
            h[e] = top;
        }
    }
};

constexpr int kKnnSeedFactor = 4;

__device__ __forceinline__ uint64_t knn_key(float d2, uint32_t id) {
    return ((uint64_t)__float_as_uint(d2) << 32) | id;
}

// The place of c in the sorted Morton codes (lower bound of its own code).
__device__ __forceinline__ int rank_of(float3 c, const uint64_t *__restrict__ codes, int n,
                                       const float *__restrict__ bounds, int bits) {
    const uint64_t qc = morton(c.x, c.y, c.z, make_grid(bounds, bits / 3));
    int lo = 0, hi = n;
    while (lo < hi) {
        const int mid = (lo + hi) >> 1;
        if (__ldg(codes + mid) < qc) lo = mid + 1;
        else hi = mid;
    }
    return lo;
}

// The k nearest primitives of one query point by one thread: Algorithm 1 with a ball
// whose radius is the current k-th best distance. The radius only shrinks
// during the walk, so a subtree the walk skips (its box farther than the
// radius then) holds no primitive that could enter the list later: the walk
// stays exact. A node is entered when its box distance is <= the radius (a
// primitive at exactly that distance may still win on its index). The list
// starts from the m = min(k, n) leaves around the query's place in the
// sorted Morton codes (a lower-bound search of the query's own code): the
// best m of the 4m leaves there, so the walk starts with a tight radius; the
// seed leaves are not considered again (a seed that left the list cannot
// come back, the radius only shrinking). 4m seeds: 16-nearest-neighbour
// walk of 2^25 uniform points 123 ms with m seeds.
// Queries with a non-finite coordinate get no neighbours. Row qi of out_idx
// / out_d2 holds the neighbours in the order (d2, index), padded with
// 0xffffffff / +inf.
template <int kP, int kCap>
__device__ __forceinline__ void heap_walk(const TreeView &t, const uint64_t *__restrict__ codes,
                                          const float *__restrict__ bounds, int bits, const QueryArgs &qa, int k,
                                          uint32_t *__restrict__ out_idx, float *__restrict__ out_d2, Control *ctl,
                                          int64_t qi) {
    const float3 c = make_float3(__ldcs(qa.queries + 3 * qi), __ldcs(qa.queries + 3 * qi + 1),
                                 __ldcs(qa.queries + 3 * qi + 2));
    const int n = (int)t.n;
    const int m = k < n ? k : n;
    KnnHeap<kCap> hp;
    hp.cnt = 0;
    const bool finite = isfinite(c.x) && isfinite(c.y) && isfinite(c.z);
    if (finite && n > 0 && ctl->build_flags == 0) {
        const int ni = n - 1;
        const float4 *base = t.inodes;  // leaves follow the internal records
        // the seed leaves [s0, s0 + S): S = 4m around the query's place in
        // Morton order (the best m of them start the list)
        const int S = min(n, kKnnSeedFactor * m);
        int s0 = 0;
        if (codes && bits > 0 && S < n) {
            s0 = min(max(rank_of(c, codes, n, bounds, bits) - S / 2, 0), n - S);
        }
        for (int j = s0; j < s0 + S; ++j) {
            const int unit = kP == LBVH_PRIM_BOXES ? 2 * (ni + j) : ni + j + ni;
            float4 a, b;
            load_node<kP>(base, unit, true, a, b);
            const uint64_t key = knn_key(box_d2(c, xyz(a), xyz(b)), __float_as_uint(a.w) & kLeafIndexMask);
            if (hp.cnt < m) hp.push(key);
            else if (key < hp.h[0]) hp.sift_from_top(key, m);
        }
        if (S < n) {
            const int nodes = 2 * n - 1;
            const uint32_t max_steps = 2u * (uint32_t)nodes;
            uint32_t steps = 0;
            int node = 0;
            while ((uint32_t)node < (uint32_t)nodes) {
                if (++steps > max_steps) break;
                const bool leaf = node >= ni;
                const int unit = kP == LBVH_PRIM_BOXES ? 2 * node : (leaf ? node + ni : 2 * node);
                float4 a, b;
                load_node<kP>(base, unit, leaf, a, b);
                const float d2 = box_d2(c, xyz(a), xyz(b));
                const uint64_t worst = hp.h[0];  // the list is full (m entries) from the seeds on
                const bool inside = d2 <= __uint_as_float((uint32_t)(worst >> 32));
                const uint32_t word = __float_as_uint(a.w);
                if (leaf) {
                    const int pos = node - ni;
                    if (inside && (pos < s0 || pos >= s0 + S)) {
                        const uint64_t key = knn_key(d2, word & kLeafIndexMask);
                        if (key < worst) hp.sift_from_top(key, m);
                    }
                    node = node + 1 - ((word & kLeafSkipInternal) ? ni : 0);
                } else {
                    node = __float_as_int(inside ? a.w : b.w);
                }
            }
            if (!(node == kSentinel || node == nodes)) atomicOr(&ctl->query_flags, kFlagCorrupt);
        }
        hp.sort();
    }
    uint32_t *ri = out_idx + qi * k;
    float *rd = out_d2 ? out_d2 + qi * k : nullptr;
    for (int r = 0; r < k; ++r) {
        const bool have = r < hp.cnt;
        const uint64_t key = have ? hp.h[r] : ~0ull;
        __stcs(ri + r, have ? (uint32_t)key : 0xffffffffu);
        if (rd) __stcs(rd + r, have ? __uint_as_float((uint32_t)(key >> 32)) : __int_as_float(0x7f800000));
    }
}

template <int kP, int kCap>
__global__ void __launch_bounds__(128)
    knn_kernel(TreeView t, const uint64_t *__restrict__ codes, const float *__restrict__ bounds, int bits,
               QueryArgs qa, int k, uint32_t *__restrict__ out_idx, float *__restrict__ out_d2, Control *ctl) {
    const int64_t i = (int64_t)blockIdx.x * 128 + threadIdx.x;
    if (i < qa.nq)
        heap_walk<kP, kCap>(t, codes, bounds, bits, qa, k, out_idx, out_d2, ctl, thread_query(qa, i));
}

// ---------------------------------------------------------------- packets

// In packets of 32 neighbouring query points, for 5 <= k <= kKnnPacketK
// (walks of n points as their own queries, heap_walk / packets, ms: 5.0M
// uniform, k = 16: 9.52 / 3.73; 2.8M of a mixture, k = 16: 6.22 / 3.21, k = 32:
// 14.5 / 6.9; 1.0M uniform, k = 8: 0.93 / 0.50; 12,001, k = 8: 0.10 / 0.10;
// k = 3: 0.4M uniform 0.19 / 0.22, 1.0M mixture 0.66 / 0.56, so fewer than 5
// stay with the heap):
//   1. knn_radius_kernel  per query an upper bound of its k-th squared
//      distance: the k-th smallest one of the kKnnMul * K leaves around its
//      place in the sorted codes (K: k rounded up to 8, 16 or 32;
//      neighbouring queries read nearly the same leaves, coalesced).
//   2. knn_packet_kernel  the ball of that radius is a range query; the
//      packet's walk keeps the hits' (distance, index) keys. A few queries
//      with a wide bound would widen the whole packet's region, so a bound is
//      cut to kKnnCut times the fourth smallest of the packet.
//   3. knn_select_kernel  a thread per query picks the k smallest keys in
//      order, by sorting networks in registers. With at least k hits they are
//      the k nearest: everything at most as far as the k-th is in the ball.
//   4. knn_redo_kernel    queries with fewer hits (their bound was cut too
//      far) or more than are kept (a bound from leaves far away),
//      8 lanes each with a bound that shrinks.
// A bound of no distance comes with an index: of many copies of a point only those
// up to it can be among the k (16 nearest of 2 * 10^6 points on 27,000 places 4.91
// ms with distances alone, so 1.11, the heap 1.19; 100,000 points on 100 places
// 1.66, 0.80, 0.61). Indices beside every bound, and equal blocks in the order of
// their leaves, cost mixtures 5 to 8%.
// Leaves of the bound's window and hits kept per query, in units of K.
template <int kK>
constexpr int kKnnMul = kK <= 8 ? 8 : 4;
template <int kK>
constexpr float kKnnCut = kK <= 8 ? 2.4f : 1.6f;
constexpr uint32_t kNoNeighbours = 0xffffffffu;  // counts[]: a query with a non-finite coordinate

template <typename T>
__device__ __forceinline__ void order2(T &a, T &b) {
    const T lo = a < b ? a : b;
    b = a ^ b ^ lo;  // a second select instead: 2.8M points, k = 32 4.45 ms, so 4.01; 5.0M, k = 16 3.80, 3.76
    a = lo;
}
template <>
__device__ __forceinline__ void order2<float>(float &a, float &b) {
    const float lo = fminf(a, b), hi = fmaxf(a, b);
    a = lo;
    b = hi;
}

// Batcher's odd-even merge sort, ascending, of kK values (a power of two); as
// templates, so that every index is a constant and the values stay in
// registers. Network<kLo, kN>: sorts v[kLo, kLo + kN); Merge: merges the two
// sorted halves of the elements kLo, kLo + kR, ... of it.
template <int kLo, int kN, int kR>
struct MergeNet {
    template <typename T, int kK>
    static __device__ __forceinline__ void run(T (&v)[kK]) {
        constexpr int m = 2 * kR;
        if constexpr (m < kN) {
            MergeNet<kLo, kN, m>::run(v);
            MergeNet<kLo + kR, kN, m>::run(v);
#pragma unroll
            for (int i = kLo + kR; i + kR < kLo + kN; i += m) order2(v[i], v[i + kR]);
        } else {
            order2(v[kLo], v[kLo + kR]);
        }
    }
};
template <int kLo, int kN>
struct SortNet {
    template <typename T, int kK>
    static __device__ __forceinline__ void run(T (&v)[kK]) {
        if constexpr (kN > 1) {
            SortNet<kLo, kN / 2>::run(v);
            SortNet<kLo + kN / 2, kN / 2>::run(v);
            MergeNet<kLo, kN, 1>::run(v);
        }
    }
};
template <int kK, typename T>
__device__ __forceinline__ void sort_values(T (&v)[kK]) {
    SortNet<0, kK>::run(v);
}

// Sorts a bitonic v: pairs kD apart, then half that, down to neighbours.
template <int kK, int kD>
struct HalveNet {
    template <typename T>
    static __device__ __forceinline__ void run(T (&v)[kK]) {
        if constexpr (kD >= 1) {
#pragma unroll
            for (int i = 0; i < kK; ++i)
                if ((i & kD) == 0) order2(v[i], v[i | kD]);
            HalveNet<kK, kD / 2>::run(v);
        }
    }
};
template <int kK>
struct HalveNet<kK, 0> {
    template <typename T>
    static __device__ __forceinline__ void run(T (&)[kK]) {}
};

// best: the kK smallest of best and v (both ascending), ascending: the
// element-wise minimum of best and v reversed is bitonic and holds them.
template <int kK, typename T>
__device__ __forceinline__ void merge_smallest(T (&best)[kK], const T (&v)[kK]) {
#pragma unroll
    for (int i = 0; i < kK; ++i) best[i] = best[i] < v[kK - 1 - i] ? best[i] : v[kK - 1 - i];
    HalveNet<kK, kK / 2>::run(best);
}

template <int kP>
__device__ __forceinline__ float leaf_d2(const float4 *leaves, int64_t pos, float3 c) {
    if (kP == LBVH_PRIM_BOXES) {
        float4 a, b;
        ld_node32(leaves + 2 * pos, a, b);
        return box_d2(c, xyz(a), xyz(b));
    }
    const float3 p = xyz(__ldg(leaves + pos));
    return box_d2(c, p, p);
}

// radii2[j]: the bound of the query at walk position first + j, NaN for one
// with a non-finite coordinate. `own`: the queries are the tree's primitives
// in sorted order, so a walk position is a place in the codes. ids[j], only where
// the bound is 0 (copies of a point, boxes around it): the largest index of k
// of those leaves that lie at no distance, which ties at the bound need not exceed.
template <int kP, int kK>
__global__ void __launch_bounds__(128)
    knn_radius_kernel(TreeView t, const uint64_t *__restrict__ codes, const float *__restrict__ bounds, int bits,
                      QueryArgs qa, int k, int64_t first, int64_t count, bool own, float *__restrict__ radii2,
                      uint32_t *__restrict__ ids, const Control *ctl) {
    const int64_t j = (int64_t)blockIdx.x * 128 + threadIdx.x;
    if (j >= count || ctl->build_flags != 0) return;
    const int64_t qi = thread_query(qa, first + j);
    const float3 c = make_float3(__ldg(qa.queries + 3 * qi), __ldg(qa.queries + 3 * qi + 1), __ldg(qa.queries + 3 * qi + 2));
    const int n = (int)t.n;
    float bound = __int_as_float(0x7fffffff);
    if (isfinite(c.x) && isfinite(c.y) && isfinite(c.z)) {
        const int rank = own ? (int)(first + j) : rank_of(c, codes, n, bounds, bits);
        constexpr int kMul = kKnnMul<kK>;
        const int s0 = min(max(rank - kMul / 2 * kK, 0), n - kMul * kK);  // n >= kMul kK
        float best[kK], v[kK];
#pragma unroll
        for (int i = 0; i < kK; ++i) best[i] = leaf_d2<kP>(t.leaves, s0 + i, c);
        sort_values(best);
#pragma unroll 1
        for (int g = 1; g < kMul; ++g) {
#pragma unroll
            for (int i = 0; i < kK; ++i) v[i] = leaf_d2<kP>(t.leaves, s0 + g * kK + i, c);
            sort_values(v);
            merge_smallest(best, v);
        }
#pragma unroll
        for (int i = 0; i < kK; ++i)
            if (i == k - 1) bound = best[i];
        if (bound == 0.0f) {
            uint32_t id = 0;
            for (int i = s0, left = k; left > 0; ++i)  // k of the window's kMul kK leaves
                if (leaf_d2<kP>(t.leaves, i, c) == 0.0f) {
                    id = max(id, __float_as_uint(t.leaves[kP == LBVH_PRIM_BOXES ? 2 * (int64_t)i : i].w) & kLeafIndexMask);
                    --left;
                }
            ids[j] = id;
        }
    }
    radii2[j] = bound;
}

// A lane's hits with their squared distances: (index, distance) words, the
// first kCap of them kept, two per 16-byte store. kCopies: `last` is looked at.
template <int kCap, bool kCopies>
struct KnnKeeper {
    // Several times what a packet reads (about 180 leaf blocks for k = 16):
    // a few queries far out, whose wide balls reach into a dense part, kept
    // one warp busy for 2 ms on a mixture of 2.8M points.
    static constexpr int kMaxBlocks = 128 + 4 * kCap;
    uint2 *slot;
    float3 c;
    uint32_t last;  // the largest index that counts
    uint32_t cnt;
    uint2 held;
    __device__ __forceinline__ bool full() const { return cnt > (uint32_t)kCap; }
    __device__ __forceinline__ void reset() { cnt = 0; }
    template <int kP, typename Q>
    __device__ __forceinline__ void take(uint32_t m, const PacketSmem<kP> &sm, int ring, const Q &) {
        if (kCopies && last != ~0u)
            for (uint32_t r = m; r; r &= r - 1) {
                const int b = 31 - __clz(r & (0u - r));
                if (sm.id[ring + 31 - b] > last) m ^= 1u << b;
            }
        const bool over = cnt + __popc(m) > (uint32_t)kCap;  // the slot is filled up, the rest dropped
        if (over)
            while (m && cnt + __popc(m) > (uint32_t)kCap) m &= m - 1;
        while (m) {
            const int b = 31 - __clz(m);
            m ^= 1u << b;
            const int at = ring + 31 - b;
            const float3 lo = make_float3(sm.cand[0][at], sm.cand[1][at], sm.cand[2][at]);
            const float3 hi = kP == LBVH_PRIM_POINTS
                                  ? lo
                                  : make_float3(sm.cand[PacketSmem<kP>::kDim - 3][at], sm.cand[PacketSmem<kP>::kDim - 2][at],
                                                sm.cand[PacketSmem<kP>::kDim - 1][at]);
            const uint2 e = make_uint2(sm.id[at], __float_as_uint(box_d2(c, lo, hi)));
            if (cnt & 1u) *reinterpret_cast<uint4 *>(slot + cnt - 1) = make_uint4(held.x, held.y, e.x, e.y);
            held = e;
            ++cnt;
        }
        if (over) cnt = kCap + 1;
    }
};

template <int kP, int kK>
__global__ void __launch_bounds__(32 * kPacketWarps, kPacketCtas<kP>)
    knn_packet_kernel(const float4 *__restrict__ leaves, const float4 *__restrict__ rec, int n, uint32_t start0,
                      QueryArgs qa, int64_t first, int64_t count, const float *__restrict__ radii2,
                      const uint32_t *__restrict__ ids, uint2 *__restrict__ slots, uint32_t *__restrict__ counts, const Control *ctl) {
    constexpr int kCap = kKnnMul<kK> * kK;
    __shared__ PacketSmem<kP> s_all[kPacketWarps];
    PacketSmem<kP> &sm = s_all[threadIdx.x >> 5];
    const int lane = threadIdx.x & 31;
    const int64_t w = (int64_t)blockIdx.x * kPacketWarps + (threadIdx.x >> 5);
    const int64_t j = w * 32 + lane;
    if (w * 32 >= count || ctl->build_flags != 0) return;
    const bool has = j < count;
    const int64_t qi = has ? thread_query(qa, first + j) : 0;
    Sphere q{make_float3(0.f, 0.f, 0.f), __int_as_float(0x7fffffff)};
    if (has)
        q = Sphere{make_float3(__ldg(qa.queries + 3 * qi), __ldg(qa.queries + 3 * qi + 1), __ldg(qa.queries + 3 * qi + 2)),
                   radii2[j]};
    const bool finite = !isnan(q.r2);
    // the fourth smallest bound of the packet (of equal ones, any)
    const float inf = __int_as_float(0x7f800000);
    float rest = has && finite ? q.r2 : inf, fourth = inf;
#pragma unroll
    for (int r = 0; r < 4; ++r) {
        const float least = warp_min(rest);
        if (least < inf) fourth = least;
        const uint32_t same = __ballot_sync(kFull, rest == least);
        if (lane == __ffs(same) - 1) rest = inf;
    }
    const bool copies = has && q.r2 == 0.0f;  // bounded by an index as well
    if (finite) q.r2 = fminf(q.r2, kKnnCut<kK> * fourth);
    const auto walk = [&](auto k) {
        const uint32_t left =
            packets<LBVH_Q_SPHERE, kP>(Blocks{leaves, rec, n, start0}, sm, q, __ballot_sync(kFull, has), k);
        if (!has) return;
        if (k.cnt <= (uint32_t)kCap && (k.cnt & 1u)) k.slot[k.cnt - 1] = k.held;
        counts[j] = !finite ? kNoNeighbours : ((left >> lane) & 1u) ? 0u : k.cnt;
    };
    if (!__any_sync(kFull, copies)) {
        walk(KnnKeeper<kCap, false>{slots + j * kCap, q.c, ~0u, 0u, make_uint2(0u, 0u)});
    } else {
        walk(KnnKeeper<kCap, true>{slots + j * kCap, q.c, copies ? ids[j] : ~0u, 0u, make_uint2(0u, 0u)});
    }
}

// Sorts the cnt keys of a query (8 lanes, kCap keys of shared memory at most)
// and keeps the first k: every key's place is the number of smaller ones (the
// keys are distinct). Returns the number kept. Called by whole warps.
template <int kCap>
__device__ __forceinline__ int keep_smallest(uint64_t *keys, int cnt, int k, int sl) {
    uint64_t mine[kCap / 8];
    int place[kCap / 8];
#pragma unroll
    for (int i = 0; i < kCap / 8; ++i) {
        mine[i] = sl + 8 * i < cnt ? keys[sl + 8 * i] : ~0ull;
        place[i] = 0;
    }
    for (int f = 0; f < cnt; ++f) {
        const uint64_t other = keys[f];
#pragma unroll
        for (int i = 0; i < kCap / 8; ++i) place[i] += other < mine[i];
    }
    __syncwarp();
#pragma unroll
    for (int i = 0; i < kCap / 8; ++i)
        if (sl + 8 * i < cnt && place[i] < k) keys[place[i]] = mine[i];
    __syncwarp();
    return min(cnt, k);
}

// The queries of `redo`, 8 lanes each through the leaf blocks (as
// sparse_walk; they are too few and too far apart for packets), to the end:
// the hits' keys are gathered in shared memory, cut back to the k smallest
// whenever they could overrun, and the k-th of those is the new bound. A fixed
// grid strides over the list (redo null: over all queries).
template <int kP, int kK>
__global__ void __launch_bounds__(128)
    knn_redo_kernel(const float4 *__restrict__ leaves, const float4 *__restrict__ rec, int n, uint32_t start0,
                    QueryArgs qa, int k, int64_t first, int64_t count, const float *__restrict__ radii2,
                    const uint32_t *__restrict__ ids, const uint32_t *__restrict__ redo, const uint32_t *redo_count, uint32_t *__restrict__ out_idx,
                    float *__restrict__ out_d2, const Control *ctl) {
    constexpr int kCap = kKnnMul<kK> * kK;
    __shared__ uint32_t s_stack[128 / 8][kSparseStack];
    __shared__ uint64_t s_keys[128 / 8][kCap];
    uint32_t *stack = s_stack[threadIdx.x >> 3];
    uint64_t *keys = s_keys[threadIdx.x >> 3];
    const int lane = threadIdx.x & 31, sl = lane & 7, shift = lane & 24;
    const uint32_t below = (1u << sl) - 1u;
    const int64_t total = redo ? min((int64_t)*redo_count, count) : count;
    const bool built = ctl->build_flags == 0;
    const int64_t stride = ((int64_t)gridDim.x * 128) >> 5;
    for (int64_t g = ((int64_t)blockIdx.x * 128 + threadIdx.x) >> 5; 4 * g < total; g += stride) {
        const bool go = 4 * g + (lane >> 3) < total;
        const int64_t j = !go ? 0 : redo ? redo[4 * g + (lane >> 3)] : 4 * g + (lane >> 3);
        const int64_t qi = thread_query(qa, first + j);
        const float3 c =
            make_float3(__ldg(qa.queries + 3 * qi), __ldg(qa.queries + 3 * qi + 1), __ldg(qa.queries + 3 * qi + 2));
        float r2 = radii2[j];
        const bool copies = r2 == 0.0f;
        const uint32_t last = copies ? ids[j] : ~0u;  // the k smallest keys have no larger index
        int cnt = 0, ns = go && built ? 1 : 0;
        if (sl == 0) stack[0] = 0u;
        __syncwarp();
        while (__any_sync(kFull, ns > 0)) {
            const bool act = ns > 0;
            const uint32_t item = act ? stack[ns - 1] : 0u;
            const bool leaf = item >= start0;
            const uint32_t child = (leaf ? (item - start0) * kFan : item * kFan + 1u) + sl;
            bool hit = false;
            uint64_t key = 0;
            float d2 = 0.0f;
            if (act && !(leaf && child >= (uint32_t)n)) {
                float4 a, b;
                if (kP == LBVH_PRIM_BOXES) {
                    ld_node32((leaf ? leaves : rec) + 2 * (int64_t)child, a, b);
                } else {
                    const float4 *p = leaf ? leaves + child : rec + 2 * (int64_t)child;
                    a = __ldg(p);
                    b = a;
                    if (!leaf) b = __ldg(p + 1);
                }
                d2 = box_d2(c, xyz(a), xyz(b));
                hit = d2 <= r2 && (leaf || __float_as_uint(b.w) == kBlockExists);
                key = knn_key(d2, __float_as_uint(a.w) & kLeafIndexMask);
                if (copies && leaf && (uint32_t)key > last) hit = false;
            }
            const uint32_t bits = (__ballot_sync(kFull, hit) >> shift) & 0xffu;
            if (act) --ns;
            __syncwarp();  // every lane has read its item
            uint32_t before = (uint32_t)__popc(bits & below);
            if (__any_sync(kFull, !leaf && __popc(bits) > 1)) {  // the nearest block on top: the bound shrinks sooner
                const float far = hit ? d2 : -1.0f;
                uint32_t farther = 0;
#pragma unroll
                for (int o = 1; o < kFan; ++o) {
                    const float other = __shfl_xor_sync(kFull, far, o);
                    farther += other > far || (other == far && (sl ^ o) < sl);
                }
                if (!leaf) before = farther;
            }
            if (!leaf) {
                if (hit) stack[ns + before] = child;
                ns += __popc(bits);
            } else {
                if (hit) keys[cnt + before] = key;
                cnt += __popc(bits);
            }
            __syncwarp();
            if (__any_sync(kFull, cnt > kCap - 8)) {
                const int kept = keep_smallest<kCap>(keys, cnt > kCap - 8 ? cnt : 0, k, sl);
                if (cnt > kCap - 8) {
                    cnt = kept;
                    r2 = fminf(r2, __uint_as_float((uint32_t)(keys[k - 1] >> 32)));
                }
                __syncwarp();
            }
        }
        cnt = keep_smallest<kCap>(keys, cnt, k, sl);
        if (go)
            for (int r = sl; r < k; r += 8) {
                out_idx[qi * k + r] = r < cnt ? (uint32_t)keys[r] : 0xffffffffu;
                if (out_d2)
                    out_d2[qi * k + r] = r < cnt ? __uint_as_float((uint32_t)(keys[r] >> 32)) : __int_as_float(0x7f800000);
            }
        __syncwarp();  // the keys are read before the next query's
    }
}

// A query with too few or too many hits goes to the list `redo`; radii2 and ids
// hold its bound (the uncut one, or the k-th smallest of the kCap hits kept).
template <int kK>
__global__ void __launch_bounds__(128)
    knn_select_kernel(QueryArgs qa, int k, int64_t first, int64_t count, const uint2 *__restrict__ slots,
                      const uint32_t *__restrict__ counts, float *__restrict__ radii2, uint32_t *__restrict__ ids,
                      uint32_t *redo,
                      uint32_t *redo_count, uint32_t *__restrict__ out_idx, float *__restrict__ out_d2,
                      const Control *ctl) {
    constexpr int kCap = kKnnMul<kK> * kK;
    const int64_t j = (int64_t)blockIdx.x * 128 + threadIdx.x;
    if (j >= count) return;
    const int64_t qi = thread_query(qa, first + j);
    uint32_t c = ctl->build_flags != 0 ? kNoNeighbours : counts[j];
    const bool none = c == kNoNeighbours;
    if (!none && c < (uint32_t)k) {
        redo[atomicAdd(redo_count, 1u)] = (uint32_t)j;
        return;
    }
    const bool over = !none && c > (uint32_t)kCap;
    if (over) c = kCap;
    if (none) c = 0;
    const uint4 *src = reinterpret_cast<const uint4 *>(slots + j * kCap);
    uint64_t best[kK], v[kK];
    auto load = [&](uint64_t (&to)[kK], int g) {
#pragma unroll
        for (int i = 0; i < kK; i += 2) {
            const uint32_t at = (uint32_t)(g * kK + i);
            uint4 e = make_uint4(~0u, ~0u, ~0u, ~0u);
            if (at < c) e = src[at / 2];
            to[i] = at < c ? (uint64_t)e.y << 32 | e.x : ~0ull;
            to[i + 1] = at + 1 < c ? (uint64_t)e.w << 32 | e.z : ~0ull;
        }
        sort_values(to);
    };
    load(best, 0);
#pragma unroll 1
    for (int g = 1; g < kKnnMul<kK> && __any_sync(__activemask(), (uint32_t)(g * kK) < c); ++g) {
        load(v, g);
        merge_smallest(best, v);
    }
    if (over) {  // the k-th smallest of some hits bounds the k-th of all
        uint64_t bound = 0;
#pragma unroll
        for (int i = 0; i < kK; ++i)
            if (i == k - 1) bound = best[i];
        radii2[j] = __uint_as_float((uint32_t)(bound >> 32));
        if (bound >> 32 == 0) ids[j] = (uint32_t)bound;
        redo[atomicAdd(redo_count, 1u)] = (uint32_t)j;
        return;
    }
    uint32_t *ri = out_idx + qi * k;
    float *rd = out_d2 ? out_d2 + qi * k : nullptr;
    const bool vec = k == kK && (reinterpret_cast<uintptr_t>(out_idx) & 15u) == 0 &&
                     (reinterpret_cast<uintptr_t>(out_d2) & 15u) == 0 && !none;
    if (vec) {
#pragma unroll
        for (int i = 0; i < kK; i += 4) {
            __stcs(reinterpret_cast<uint4 *>(ri + i), make_uint4((uint32_t)best[i], (uint32_t)best[i + 1],
                                                                 (uint32_t)best[i + 2], (uint32_t)best[i + 3]));
            if (rd)
                __stcs(reinterpret_cast<uint4 *>(rd + i),
                       make_uint4((uint32_t)(best[i] >> 32), (uint32_t)(best[i + 1] >> 32), (uint32_t)(best[i + 2] >> 32),
                                  (uint32_t)(best[i + 3] >> 32)));
        }
        return;
    }
#pragma unroll
    for (int i = 0; i < kK; ++i) {
        if (i >= k) break;
        ri[i] = none ? 0xffffffffu : (uint32_t)best[i];
        if (rd) rd[i] = none ? __int_as_float(0x7f800000) : __uint_as_float((uint32_t)(best[i] >> 32));
    }
}

}  // namespace

void launch_knn(const TreeView &t, const uint64_t *codes, const float *bounds, int bits, const QueryArgs &q, int k,
                uint32_t *out_idx, float *out_d2, Control *ctl, cudaStream_t s) {
    if (q.nq <= 0) return;
    const unsigned blocks = (unsigned)((q.nq + 127) / 128);
    auto go = [&](auto cap) {
        constexpr int C = decltype(cap)::value;
        if (t.kind == LBVH_PRIM_POINTS)
            knn_kernel<LBVH_PRIM_POINTS, C><<<blocks, 128, 0, s>>>(t, codes, bounds, bits, q, k, out_idx, out_d2, ctl);
        else
            knn_kernel<LBVH_PRIM_BOXES, C><<<blocks, 128, 0, s>>>(t, codes, bounds, bits, q, k, out_idx, out_d2, ctl);
    };
    if (k <= 16) go(std::integral_constant<int, 16>{});
    else if (k <= 64) go(std::integral_constant<int, 64>{});
    else go(std::integral_constant<int, kKnnMaxK>{});
    count_launches(1);
}


namespace {

int knn_class(int k) { return k <= 8 ? 8 : k <= 16 ? 16 : 32; }

template <int kP, int kK>
void knn_chunks(const TreeView &t, const float4 *rec, const uint64_t *codes, const float *bounds, int bits,
                const QueryArgs &q, bool own, int k, KnnWalk how, const KnnScratch &sc, uint32_t *out_idx, float *out_d2,
                Control *ctl, cudaStream_t s) {
    const int64_t redo_grid = (int64_t)device_sm_count() * 12;
    if (how == kKnnSparse) {  // one chunk: the bounds, then 8 lanes for every query
        knn_radius_kernel<kP, kK><<<(unsigned)((q.nq + 127) / 128), 128, 0, s>>>(t, codes, bounds, bits, q, k, 0, q.nq, own,
                                                                                 sc.radii2, sc.ids, ctl);
        knn_redo_kernel<kP, kK><<<(unsigned)std::min<int64_t>((q.nq + 15) / 16, redo_grid), 128, 0, s>>>(
            t.leaves, rec, (int)t.n, pack_leaf_start(t.n), q, k, 0, q.nq, sc.radii2, sc.ids, nullptr, nullptr, out_idx, out_d2, ctl);
        count_launches(2);
        return;
    }
    cudaMemsetAsync(sc.redo_counts, 0, (size_t)((q.nq + sc.chunk - 1) / sc.chunk) * 4, s);
    const uint32_t start0 = pack_leaf_start(t.n);
    for (int64_t first = 0; first < q.nq; first += sc.chunk) {
        const int64_t count = std::min(sc.chunk, q.nq - first);
        const unsigned blocks = (unsigned)((count + 127) / 128);
        knn_radius_kernel<kP, kK><<<blocks, 128, 0, s>>>(t, codes, bounds, bits, q, k, first, count, own, sc.radii2, sc.ids,
                                                      ctl);
        knn_packet_kernel<kP, kK><<<(unsigned)((count + 32 * kPacketWarps - 1) / (32 * kPacketWarps)), 32 * kPacketWarps, 0,
                                    s>>>(t.leaves, rec, (int)t.n, start0, q, first, count, sc.radii2, sc.ids, sc.slots, sc.counts,
                                         ctl);
        uint32_t *redo_count = sc.redo_counts + first / sc.chunk;
        knn_select_kernel<kK><<<blocks, 128, 0, s>>>(q, k, first, count, sc.slots, sc.counts, sc.radii2, sc.ids, sc.redo, redo_count,
                                                     out_idx, out_d2, ctl);
        knn_redo_kernel<kP, kK><<<(unsigned)std::min<int64_t>((count + 15) / 16, redo_grid), 128, 0,
                                  s>>>(t.leaves, rec, (int)t.n, start0, q, k, first, count, sc.radii2, sc.ids, sc.redo, redo_count,
                                       out_idx, out_d2, ctl);
        count_launches(4);
    }
}

}  // namespace

// 8 lanes per query against the heap (its query order included; us): 100,003
// uniform points, 10,000 queries, k = 3: 57 / 127, k = 32: 143 / 406;
// 3.0M points, 30,000 queries, k = 3: 114 / 152, k = 16: 179 / 427; 77,000
// queries, k = 3: 229 / 193, k = 16: 389 / 519; 150,000, k = 16: about equal.
// 9,001 points as their own queries (the order is free), k = 1: 31 / 18, k = 3:
// 47 / 57.
KnnWalk knn_walk(int64_t nq, int64_t n, int k, bool sorted) {
    const int64_t sms = device_sm_count();
    if (k > kKnnPacketK || n < 1024) return kKnnHeap;
    const bool dense = n <= 4 * nq;
    if (k >= 5 && dense && nq >= 64 * sms) return kKnnPackets;
    const int64_t few = k <= 2 && sorted ? 0 : dense ? 64 : k >= 5 ? 512 : 256;
    return nq <= few * sms ? kKnnSparse : kKnnHeap;
}

int64_t knn_chunk(int64_t nq) { return std::min<int64_t>(nq, int64_t(1) << 20); }
size_t knn_slot_bytes(int k) { return (size_t)(k <= 8 ? 8 : 4) * knn_class(k) * sizeof(uint2); }

void launch_knn_packets(const TreeView &t, const float4 *rec, const uint64_t *codes, const float *bounds, int bits,
                        const QueryArgs &q, bool own, int k, KnnWalk how, const KnnScratch &sc, uint32_t *out_idx,
                        float *out_d2, Control *ctl, cudaStream_t s) {
    if (q.nq <= 0) return;
    auto go = [&](auto kk) {
        constexpr int K = decltype(kk)::value;
        if (t.kind == LBVH_PRIM_POINTS)
            knn_chunks<LBVH_PRIM_POINTS, K>(t, rec, codes, bounds, bits, q, own, k, how, sc, out_idx, out_d2, ctl, s);
        else
            knn_chunks<LBVH_PRIM_BOXES, K>(t, rec, codes, bounds, bits, q, own, k, how, sc, out_idx, out_d2, ctl, s);
    };
    switch (knn_class(k)) {
    case 8: go(std::integral_constant<int, 8>{}); break;
    case 16: go(std::integral_constant<int, 16>{}); break;
    default: go(std::integral_constant<int, 32>{}); break;
    }
}

}  // namespace lbvh
