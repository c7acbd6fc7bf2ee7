// packet.cu -- range queries by packets over leaf blocks.
//
// Algorithm 1 visits the nodes of one query's path one after the other: about
// 170 dependent loads for the 16 hits of a query among 2^25 uniform points, of
// which 140 are internal nodes. Neighbouring queries visit nearly the same
// ones. Here a warp answers 32 neighbouring queries (a packet) together, over
// a second, implicit tree: the sorted leaves cut into blocks of 8, the blocks
// into blocks of 8, and so on, each with its box (see launch_pack). The 8
// children of a block are 8 consecutive records, so a step of a walk reads
// them coalesced, one per lane, and needs no topology.
//
// packet_kernel  a warp per 32 walk positions.
//   1. The packet's region: what every query of the packet lies in (the box
//      of the centres and the largest radius; the union of the query boxes).
//      Its test against a box is computed with the operations of the single
//      test, each of which is monotone, so it holds wherever one of the
//      queries' own tests holds.
//   2. Blocks are taken from a stack in shared memory, four at a time, their
//      32 children tested against the region, those that pass pushed; leaf
//      blocks go to a list.
//   3. Leaf blocks are read four at a time (32 leaves), the leaves that meet
//      the region go to a candidate buffer, and every 32 candidates are
//      tested by every lane against its own query with the exact predicate,
//      the candidates' coordinates broadcast from shared memory.
// sparse_kernel  8 lanes per query: the lanes test the 8 children of one
//   block at a time with the query's own predicate. For few queries and few
//   rays (more warps in flight, a shorter chain of loads, no query order to
//   compute). Packets whose queries lie too far apart for a common region are
//   left to collect_left_kernel (query.cu).
//
// Both report exactly the primitives whose own test holds, like Algorithm 1
// (the hit lists are sorted afterwards, so their order here does not matter).
#include <algorithm>
#include <type_traits>

#include "lbvh_internal.cuh"
#include "packet.cuh"
#include "walk.cuh"

namespace lbvh {

namespace {

// ---------------------------------------------------------------- boxes of the leaf blocks

struct Bounds {
    float3 lo, hi;
};

__device__ __forceinline__ Bounds empty_bounds() {
    const float inf = __int_as_float(0x7f800000);
    return Bounds{make_float3(inf, inf, inf), make_float3(-inf, -inf, -inf)};
}

__device__ __forceinline__ void grow(Bounds &b, const Bounds &o) {
    b.lo = make_float3(fminf(b.lo.x, o.lo.x), fminf(b.lo.y, o.lo.y), fminf(b.lo.z, o.lo.z));
    b.hi = make_float3(fmaxf(b.hi.x, o.hi.x), fmaxf(b.hi.y, o.hi.y), fmaxf(b.hi.z, o.hi.z));
}

__device__ __forceinline__ Bounds xor_lane(const Bounds &b, int off) {
    Bounds o;
    o.lo.x = __shfl_xor_sync(kFull, b.lo.x, off);
    o.lo.y = __shfl_xor_sync(kFull, b.lo.y, off);
    o.lo.z = __shfl_xor_sync(kFull, b.lo.z, off);
    o.hi.x = __shfl_xor_sync(kFull, b.hi.x, off);
    o.hi.y = __shfl_xor_sync(kFull, b.hi.y, off);
    o.hi.z = __shfl_xor_sync(kFull, b.hi.z, off);
    return o;
}

// A record: the box, and in the last word whether the block exists (levels are
// padded to a multiple of 8 records with blocks that do not).
__device__ __forceinline__ void put_block(float4 *rec, int64_t at, const Bounds &b, bool exists) {
    rec[2 * at] = make_float4(b.lo.x, b.lo.y, b.lo.z, 0.0f);
    rec[2 * at + 1] = make_float4(b.hi.x, b.hi.y, b.hi.z, __uint_as_float(exists ? kBlockExists : 0u));
}

__device__ __forceinline__ Bounds get_block(const float4 *rec, int64_t at) {
    const float4 a = __ldcg(rec + 2 * at), b = __ldcg(rec + 2 * at + 1);
    return Bounds{make_float3(a.x, a.y, a.z), make_float3(b.x, b.y, b.z)};
}

// Blocks of height h (0: leaf blocks) of a tree of n leaves, and the same
// with the padding (the root has none).
__device__ __forceinline__ int64_t blocks_of(int64_t n, int h) { return (n - 1) / ((int64_t)kFan << (3 * h)) + 1; }
__device__ __forceinline__ int64_t padded_of(int64_t n, int h, int depth) {
    return h >= depth ? 1 : (blocks_of(n, h) + kFan - 1) / kFan * kFan;
}
// The first record of height h: heap order, the root first.
__device__ __forceinline__ int64_t start_of(int h, int depth) { return ((1ll << (3 * (depth - h))) - 1) / 7; }

// The heights above `from` (and the padding of `from`), by one CTA, from the
// records of height `from`.
__device__ __forceinline__ void pack_top(int64_t n, int depth, int from, float4 *rec) {
    if (depth <= from) return;
    for (int64_t i = blocks_of(n, from) + threadIdx.x; i < padded_of(n, from, depth); i += blockDim.x)
        put_block(rec, start_of(from, depth) + i, empty_bounds(), false);
    for (int h = from + 1; h <= depth; ++h) {
        const int64_t below = blocks_of(n, h - 1), count = blocks_of(n, h), s1 = start_of(h - 1, depth);
        for (int64_t i = threadIdx.x; i < padded_of(n, h, depth); i += blockDim.x) {
            Bounds b = empty_bounds();
            for (int64_t k = kFan * i; k < min(below, kFan * (i + 1)); ++k) grow(b, get_block(rec, s1 + k));
            put_block(rec, start_of(h, depth) + i, b, i < count);
        }
        __syncthreads();
    }
}

// The CTA that takes the last of `total` tickets (all of its threads get the
// answer); the others' records are complete for it.
__device__ __forceinline__ bool last_of(uint32_t *ticket, uint32_t total) {
    __shared__ bool s_last;
    __syncthreads();
    if (threadIdx.x == 0) {
        __threadfence();
        const uint32_t t = atomicAdd(ticket, 1u);
        s_last = t == total - 1;
        if (s_last) *ticket = 0;  // ready for the next tree
    }
    __syncthreads();
    if (s_last) __threadfence();
    return s_last;
}

constexpr int kPackThreads = 128;
constexpr int kPackWarps = kPackThreads / 32;
constexpr int kPackSpan = 4096;  // leaves per CTA: one block of height 3
constexpr int kPackStep = 256;   // leaves per step of a warp: a leaf block per lane

// Points on their way to the lanes that reduce them: read 32 at a time, kept
// as rows of 8 with one more slot per row, so that the lanes' reads of their
// own rows fall into different banks. (A lane reads its 8 boxes itself: whole
// sectors either way.)
template <int kP>
struct PackSmem {
    float4 leaf[kP == LBVH_PRIM_POINTS ? kPackWarps : 1][kP == LBVH_PRIM_POINTS ? 32 * (kFan + 1) : 1];
    Bounds part[kPackWarps];
};

// Heights 0..3 of the blocks over leaves [first, first + kPackSpan) of a tree
// of n leaves (first a multiple of kPackSpan), by one CTA. What bounds it is
// memory (20 bytes per point): 0.126 ms at 2^25 points, 5.3 TB/s. With the
// lanes on consecutive leaves and shuffles over the 8 of a block it took
// 0.21 ms, issuing 3 times the instructions.
template <int kP>
__device__ __forceinline__ void pack_span(const float4 *__restrict__ leaves, int64_t n, int64_t first, int depth,
                                          float4 *rec, PackSmem<kP> &sm) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int64_t base = first + (int64_t)warp * (kPackSpan / kPackWarps);
    const int64_t pad0 = padded_of(n, 0, depth), pad1 = padded_of(n, 1, depth), pad2 = padded_of(n, 2, depth);
    Bounds two = empty_bounds(), all = empty_bounds();
    for (int k = 0; k < kPackSpan / kPackWarps / kPackStep; ++k) {
        const int64_t p0 = base + kPackStep * k;
        Bounds b = empty_bounds();
        const int64_t pos = p0 + kFan * lane;
        if constexpr (kP == LBVH_PRIM_POINTS) {
#pragma unroll
            for (int j = 0; j < kPackStep / 32; ++j) {
                const int at = 32 * j + lane;
                if (p0 + at < n) sm.leaf[warp][at + at / kFan] = __ldg(leaves + p0 + at);
            }
            __syncwarp();
#pragma unroll
            for (int j = 0; j < kFan; ++j)
                if (pos + j < n) {
                    const float3 v = xyz(sm.leaf[warp][(kFan + 1) * lane + j]);
                    grow(b, Bounds{v, v});
                }
            __syncwarp();  // the rows are rewritten by the next step
        } else {
#pragma unroll
            for (int j = 0; j < kFan; ++j)
                if (pos + j < n) {
                    float4 u, v;
                    ld_node32(leaves + 2 * (pos + j), u, v);
                    grow(b, Bounds{leaf_lo<kP>(u, v), leaf_hi<kP>(u, v)});
                }
        }
        if (pos / kFan < pad0) put_block(rec, start_of(0, depth) + pos / kFan, b, pos < n);
        for (int off = 1; off < kFan; off <<= 1) grow(b, xor_lane(b, off));
        if (lane % kFan == 0 && depth >= 1 && pos / (kFan * kFan) < pad1)
            put_block(rec, start_of(1, depth) + pos / (kFan * kFan), b, pos < n);
        for (int off = kFan; off < 32; off <<= 1) grow(b, xor_lane(b, off));
        grow(two, b);
        if (k & 1) {
            const int64_t p2 = p0 - kPackStep, at = p2 / (kFan * kFan * kFan);
            if (lane == 0 && depth >= 2 && at < pad2) put_block(rec, start_of(2, depth) + at, two, p2 < n);
            grow(all, two);
            two = empty_bounds();
        }
    }
    if (lane == 0) sm.part[warp] = all;
    __syncthreads();
    if (threadIdx.x == 0 && depth >= 3 && first < n) {
        Bounds b = sm.part[0];
        for (int w = 1; w < kPackWarps; ++w) grow(b, sm.part[w]);
        put_block(rec, start_of(3, depth) + first / kPackSpan, b, true);
    }
}

template <int kP>
__global__ void __launch_bounds__(kPackThreads)
    pack_kernel(const float4 *__restrict__ leaves, int64_t n, int depth, float4 *rec, Control *ctl) {
    __shared__ PackSmem<kP> sm;
    pack_span<kP>(leaves, n, (int64_t)blockIdx.x * kPackSpan, depth, rec, sm);
    if (depth > 3 && last_of(&ctl->pack_ticket, gridDim.x)) pack_top(n, depth, 3, rec);
}

// Batches: a CTA per chunk (two spans) of an instance, then a CTA per instance
// for the heights above 3.
template <int kP>
__global__ void __launch_bounds__(kPackThreads)
    batch_pack_kernel(const float4 *__restrict__ nodes, BatchTables bt, float4 *rec) {
    static_assert(kBatchChunk % kPackSpan == 0, "a chunk is whole spans");
    __shared__ PackSmem<kP> sm;
    const BatchChunk c = bt.chunks[blockIdx.x];
    const int64_t o = bt.prim_off[c.inst], n = bt.prim_off[c.inst + 1] - o;
    const float4 *leaves = nodes + bt.node_start[c.inst] + 2 * (n - 1);
    float4 *r = rec + 2 * bt.pack_start[c.inst];
    const int depth = pack_depth(n);
    for (int64_t at = c.begin - o; at < c.end - o; at += kPackSpan) {
        pack_span<kP>(leaves, n, at, depth, r, sm);
        __syncthreads();
    }
}

__global__ void __launch_bounds__(kPackThreads) batch_pack_top_kernel(BatchTables bt, float4 *rec) {
    const int64_t n = bt.prim_off[blockIdx.x + 1] - bt.prim_off[blockIdx.x];
    if (n > 0) pack_top(n, pack_depth(n), 3, rec + 2 * bt.pack_start[blockIdx.x]);
}

// ---------------------------------------------------------------- range queries

// A lane's query in a packet: its hits so far and its spill chunk. Hits go to
// the slot four at a time (one 16-byte store; words past the count are never
// read): the slots of a packet's queries lie apart, so every store is a
// sector of its own (walk of 2^25 uniform points: 11.96 ms with single
// stores, 9.01 with pairs, 8.97 with fours, at 12 CTAs per SM each).
struct Keeper {
    static constexpr int kMaxBlocks = 0;  // every list is taken whole
    const QueryScratch &qs;
    Control *ctl;
    uint32_t *slot;
    int64_t qi;
    uint32_t cnt, cur, h0, h1, h2;  // h0, h1, h2: the last three hits
    // `id` is the next hit; the slot has room.
    __device__ __forceinline__ void keep(uint32_t id) {
        if ((cnt & 3u) == 3u) __stcs(reinterpret_cast<uint4 *>(slot + cnt - 3), make_uint4(h0, h1, h2, id));
        h0 = h1;
        h1 = h2;
        h2 = id;
        ++cnt;
    }
    // Stores the hits of the last, incomplete four.
    __device__ __forceinline__ void drain() const {
        if (cnt >= (uint32_t)kSlot) return;
        const uint32_t r = cnt & 3u;
        if (r >= 1) __stcs(slot + cnt - 1, h2);
        if (r >= 2) __stcs(slot + cnt - 2, h1);
        if (r >= 3) __stcs(slot + cnt - 3, h0);
    }
    template <int kP, typename Q>
    __device__ __forceinline__ void take(uint32_t m, const PacketSmem<kP> &sm, int ring, const Q &) {
        const uint32_t *ids = sm.id + ring + 31;
        const bool room = !__any_sync(kFull, cnt + __popc(m) > (uint32_t)kSlot);
        if (room) {
            while (m) {
                const int b = 31 - __clz(m);
                m ^= 1u << b;
                keep(ids[-b]);
            }
        } else {  // a lane's hits run past its slot
            while (m) {
                const int b = 31 - __clz(m);
                m ^= 1u << b;
                if (cnt < (uint32_t)kSlot) {
                    keep(ids[-b]);
                } else {
                    spill_put(qs, ctl, qi, cnt, ids[-b], cur);
                    ++cnt;
                }
            }
        }
    }
    __device__ __forceinline__ void finish() const {
        drain();
        __stcs(qs.counts + qi, cnt);  // streamed: keep L2 for the tree
        if (cnt > (uint32_t)kSlot)
            qs.overflow_list[atomicAdd(&ctl->overflow_filled, 1u)] =
                (uint32_t)qi | (cur != kSpillFailed ? kSpilledTag : 0u);
    }
};

template <int kQ, int kP>
__global__ void __launch_bounds__(32 * kPacketWarps, kPacketCtas<kP>)
    packet_kernel(const float4 *__restrict__ leaves, const float4 *__restrict__ rec, int n, uint32_t start0,
                  QueryArgs qa, QueryScratch qs, Control *ctl) {
    __shared__ PacketSmem<kP> s_all[kPacketWarps];
    PacketSmem<kP> &sm = s_all[threadIdx.x >> 5];
    const int lane = threadIdx.x & 31;
    const int64_t w = (int64_t)blockIdx.x * kPacketWarps + (threadIdx.x >> 5);
    const int64_t i = w * 32 + lane;
    if (w * 32 >= qa.nq) return;
    const bool has = i < qa.nq;
    const int64_t qi = has ? thread_query(qa, i) : 0;
    Keeper k{qs, ctl, qs.slots + qi * kSlot, qi, 0u, kNoChunk, 0u, 0u, 0u};
    uint32_t left = 0;
    if (ctl->build_flags == 0) {
        typename QueryOf<kQ>::type q{};
        if (has) q = QueryOf<kQ>::load(qa, qi);
        left = packets<kQ, kP>(Blocks{leaves, rec, n, start0}, sm, q, __ballot_sync(kFull, has), k);
        if (left && lane == 0) qs.sparse_list[atomicAdd(&ctl->sparse_filled, 1u)] = make_uint2((uint32_t)w, left);
    }
    if (has && !((left >> lane) & 1u)) k.finish();
}

// Batches: the same, on the tree of the queries' instance; the instances of a
// warp's queries (runs of lanes, the order being per instance) go in turn.
template <int kQ, int kP>
__global__ void __launch_bounds__(32 * kPacketWarps, kPacketCtas<kP>)
    batch_packet_kernel(const float4 *__restrict__ nodes, const float4 *__restrict__ rec, BatchTables bt, QueryArgs qa,
                        QueryScratch qs, Control *ctl) {
    __shared__ PacketSmem<kP> s_all[kPacketWarps];
    PacketSmem<kP> &sm = s_all[threadIdx.x >> 5];
    const int lane = threadIdx.x & 31;
    const int64_t w = (int64_t)blockIdx.x * kPacketWarps + (threadIdx.x >> 5);
    const int64_t i = w * 32 + lane;
    if (w * 32 >= qa.nq) return;
    const bool has = i < qa.nq;
    const int64_t qi = has ? thread_query(qa, i) : 0;
    Keeper k{qs, ctl, qs.slots + qi * kSlot, qi, 0u, kNoChunk, 0u, 0u, 0u};
    uint32_t left = 0;
    if (ctl->build_flags == 0) {
        typename QueryOf<kQ>::type q{};
        if (has) q = QueryOf<kQ>::load(qa, qi);
        const int inst = has ? instance_of(bt.query_off, bt.count, qi) : -1;
        uint32_t rest = __ballot_sync(kFull, has);
        while (rest) {
            const int b = __shfl_sync(kFull, inst, __ffs(rest) - 1);
            const uint32_t mine = __ballot_sync(kFull, inst == b);
            rest &= ~mine;
            const int64_t n = bt.prim_off[b + 1] - bt.prim_off[b];
            if (n <= 0) continue;
            const Blocks t{nodes + bt.node_start[b] + 2 * (n - 1), rec + 2 * bt.pack_start[b], (int)n, pack_leaf_start(n)};
            left |= packets<kQ, kP>(t, sm, q, mine, k);
        }
        if (left && lane == 0) qs.sparse_list[atomicAdd(&ctl->sparse_filled, 1u)] = make_uint2((uint32_t)w, left);
    }
    if (has && !((left >> lane) & 1u)) k.finish();
}

// ---------------------------------------------------------------- 8 lanes per query

constexpr int kSparseThreads = 128;
template <int kQ, int kP>
__global__ void __launch_bounds__(kSparseThreads)
    sparse_kernel(const float4 *__restrict__ leaves, const float4 *__restrict__ rec, int n, uint32_t start0,
                  QueryArgs qa, QueryScratch qs, Control *ctl) {
    __shared__ uint32_t s_stack[kSparseThreads / 8][kSparseStack];
    const int64_t i = ((int64_t)blockIdx.x * kSparseThreads + threadIdx.x) >> 3;
    const bool has = i < qa.nq, ok = ctl->build_flags == 0;
    const int64_t qi = has ? query_at<kQ>(qa, i) : 0;
    typename QueryOf<kQ>::type q{};
    if (has && ok) q = QueryOf<kQ>::load(qa, qi);
    if (has && !ok && (threadIdx.x & 7) == 0) __stcs(qs.counts + qi, 0u);
    const Blocks blocks{leaves, rec, n, start0};
    uint32_t *stack = s_stack[threadIdx.x >> 3];
    if constexpr (kQ == LBVH_Q_RAY) {  // the general test if any of the warp's rays has a parallel axis
        if (!__any_sync(kFull, q.parallel != 0)) {
            sparse_walk<kP>(blocks, stack, SlantedRay{q}, has && ok, qi, qs, ctl);
            return;
        }
    }
    sparse_walk<kP>(blocks, stack, q, has && ok, qi, qs, ctl);
}

}  // namespace

void launch_pack(const TreeView &t, float4 *rec, Control *ctl, cudaStream_t s) {
    if (t.n <= 0) return;
    const unsigned blocks = (unsigned)((t.n + kPackSpan - 1) / kPackSpan);
    auto k = t.kind == LBVH_PRIM_POINTS ? pack_kernel<LBVH_PRIM_POINTS> : pack_kernel<LBVH_PRIM_BOXES>;
    k<<<blocks, kPackThreads, 0, s>>>(t.leaves, t.n, pack_depth(t.n), rec, ctl);
    count_launches(1);
}

void launch_batch_pack(const float4 *nodes, int kind, const BatchTables &bt, float4 *rec, cudaStream_t s) {
    if (bt.nchunks <= 0) return;
    (kind == LBVH_PRIM_POINTS ? batch_pack_kernel<LBVH_PRIM_POINTS> : batch_pack_kernel<LBVH_PRIM_BOXES>)<<<
        (unsigned)bt.nchunks, kPackThreads, 0, s>>>(nodes, bt, rec);
    batch_pack_top_kernel<<<(unsigned)bt.count, kPackThreads, 0, s>>>(bt, rec);
    count_launches(2);
}

// Measured on resident trees (walk, plus the query order where one has to be
// made; us, packets / 8 lanes per query / Algorithm 1):
//   2^23 uniform points, 2^22 queries 1603 / 6512 / 2957; 2^21 1333 / 3282 /
//   1676; 2^20 1071 / 1662 / 1051; 2^18 755 / 450 / 460; 2^17 531 / 250 / 357;
//   2^15 449 / 86 / 295; mixture boxes 2^22 1708 / 7855 / 2324, 2^21 1303 /
//   3952 / 1299; 2^20 1068 / 2003 / 834; 2^18 731 / 545 / 452.
//   As many queries as points, in the points' own order: 16384 48 / 32 / 68,
//   65536 53 / 76 / 80; in another: 2^16 113 / 76 / 139. Boxes for boxes, in
//   their own order: 70,000 121 / 109 / 109, 170,000 150 / 195 / 183; in
//   another: 119,230 for 310,000 215 / 201 / 216, 130,769 for 170,000 209 /
//   211 / 216.
// So packets need a query for at least every fourth leaf (fewer lie too far
// apart to share nodes) and enough packets to fill the GPU; below about 1000
// queries per SM the 8 lanes have the shorter chain of loads, and need no
// order; in between Algorithm 1 stays.
// Rays have no packets. 8 lanes per ray against a thread (2^23 mixture boxes,
// walk and order, us): 30,000 random segments 361 / 791, 60,000 484 / 833,
// 120,000 758 / 880, 250,000 1407 / 1100, 2^20 5364 / 2656; 20,000 on
// 30,000 49 / 130, 100,000 on 200,000 249 / 252. Few rays take as long as the
// longest walk, which is shorter by blocks; many take as long as their
// instructions.
RangeWalk range_walk(int qkind, int64_t nq, int64_t n, bool sorted) {
    if (qkind == LBVH_Q_RAY) return nq <= 640 * (int64_t)device_sm_count() ? kRangeSparse : kRangeNodes;
    const bool dense = n <= 4 * nq;
    const bool boxes = qkind == LBVH_Q_BOX;
    const int64_t few = (dense ? (sorted ? (boxes ? 512 : 256) : (boxes ? 800 : 640)) : 1024) * (int64_t)device_sm_count();
    if (nq <= few) return kRangeSparse;
    return dense ? kRangePackets : kRangeNodes;
}

namespace {

template <typename F>
void dispatch_range_kinds(int qkind, int pkind, F &&f) {
    using Points = std::integral_constant<int, LBVH_PRIM_POINTS>;
    using Boxes = std::integral_constant<int, LBVH_PRIM_BOXES>;
    using SphereQ = std::integral_constant<int, LBVH_Q_SPHERE>;
    using BoxQ = std::integral_constant<int, LBVH_Q_BOX>;
    using RayQ = std::integral_constant<int, LBVH_Q_RAY>;
    if (qkind == LBVH_Q_RAY) {
        if (pkind == LBVH_PRIM_POINTS) f(RayQ{}, Points{});
        else f(RayQ{}, Boxes{});
    } else if (qkind == LBVH_Q_SPHERE) {
        if (pkind == LBVH_PRIM_POINTS) f(SphereQ{}, Points{});
        else f(SphereQ{}, Boxes{});
    } else {
        if (pkind == LBVH_PRIM_POINTS) f(BoxQ{}, Points{});
        else f(BoxQ{}, Boxes{});
    }
}

}  // namespace

void launch_query_packets(const TreeView &t, const float4 *rec, const QueryArgs &q, const QueryScratch &qs,
                          RangeWalk how, Control *ctl, cudaStream_t s) {
    if (q.nq <= 0) return;
    const uint32_t start0 = pack_leaf_start(t.n);
    const int n = (int)t.n;
    dispatch_range_kinds(q.qkind, t.kind, [&](auto qk, auto pk) {
        constexpr int Q = decltype(qk)::value, P = decltype(pk)::value;
        if (how == kRangeSparse) {
            const unsigned blocks = (unsigned)((q.nq + kSparseThreads / 8 - 1) / (kSparseThreads / 8));
            sparse_kernel<Q, P><<<blocks, kSparseThreads, 0, s>>>(t.leaves, rec, n, start0, q, qs, ctl);
        } else if constexpr (Q != LBVH_Q_RAY) {
            const unsigned blocks = (unsigned)((q.nq + 32 * kPacketWarps - 1) / (32 * kPacketWarps));
            packet_kernel<Q, P><<<blocks, 32 * kPacketWarps, 0, s>>>(t.leaves, rec, n, start0, q, qs, ctl);
        }
    });
    count_launches(1);
    if (how != kRangeSparse) launch_query_collect_left(t, rec, q, qs, ctl, s);
}

void launch_batch_packets(const float4 *nodes, int kind, const float4 *rec, const BatchTables &bt, const QueryArgs &q,
                          const QueryScratch &qs, Control *ctl, cudaStream_t s) {
    if (q.nq <= 0) return;
    const unsigned blocks = (unsigned)((q.nq + 32 * kPacketWarps - 1) / (32 * kPacketWarps));
    dispatch_range_kinds(q.qkind, kind, [&](auto qk, auto pk) {
        if constexpr (decltype(qk)::value != LBVH_Q_RAY)
            batch_packet_kernel<decltype(qk)::value, decltype(pk)::value>
                <<<blocks, 32 * kPacketWarps, 0, s>>>(nodes, rec, bt, q, qs, ctl);
    });
    count_launches(1);
    launch_batch_collect_left(nodes, kind, bt, q, qs, ctl, s);
}

}  // namespace lbvh
