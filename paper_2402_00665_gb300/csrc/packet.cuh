// packet.cuh -- the walk of a packet (a warp's 32 neighbouring queries) through
// the leaf blocks; packet.cu says how it works. Range queries (packet.cu) and k
// nearest neighbours (knn.cu) differ in what a lane keeps of its hits.
#pragma once

#include "lbvh_internal.cuh"
#include "walk.cuh"

namespace lbvh {

// A primitive's box with its bounds in order: the exact test of a box given
// the wrong way round (lo > hi) looks at either bound, so a region has to
// meet both.
template <int kP>
__device__ __forceinline__ float3 leaf_lo(float4 a, float4 b) {
    if (kP == LBVH_PRIM_POINTS) return xyz(a);
    return make_float3(fminf(a.x, b.x), fminf(a.y, b.y), fminf(a.z, b.z));
}
template <int kP>
__device__ __forceinline__ float3 leaf_hi(float4 a, float4 b) {
    if (kP == LBVH_PRIM_POINTS) return xyz(b);
    return make_float3(fmaxf(a.x, b.x), fmaxf(a.y, b.y), fmaxf(a.z, b.z));
}

// ---------------------------------------------------------------- regions

// The region of a packet: meets() holds wherever hits() holds for one of the
// packet's queries (every operation is monotone in the query's bounds under
// round-to-nearest, so this needs no margin).
template <typename Q>
struct Region;

__device__ __forceinline__ float warp_min(float v) {
    float r;
    asm volatile("redux.sync.min.f32 %0, %1, 0xffffffff;" : "=f"(r) : "f"(v));
    return r;
}
__device__ __forceinline__ float warp_max(float v) {
    float r;
    asm volatile("redux.sync.max.f32 %0, %1, 0xffffffff;" : "=f"(r) : "f"(v));
    return r;
}

template <>
struct Region<Sphere> {
    float3 lo, hi;  // the box of the centres
    float r2;       // the largest squared radius
    static constexpr bool kShapes = false;
    // `use`: this lane's query belongs to the packet (warp-wide call)
    __device__ __forceinline__ void gather(const Sphere &s, bool use) {
        const float inf = __int_as_float(0x7f800000);
        lo = make_float3(warp_min(use ? s.c.x : inf), warp_min(use ? s.c.y : inf), warp_min(use ? s.c.z : inf));
        hi = make_float3(warp_max(use ? s.c.x : -inf), warp_max(use ? s.c.y : -inf), warp_max(use ? s.c.z : -inf));
        r2 = warp_max(use ? s.r2 : 0.0f);
    }
    // A query that can hit nothing (it would only blow the region up).
    static __device__ __forceinline__ bool hopeless(const Sphere &s) {
        return isnan(s.c.x) || isnan(s.c.y) || isnan(s.c.z) || isnan(s.r2);
    }
    // The queries overlap enough that the region is not much more than one
    // query's own: the centres spread over at most 4 radii.
    __device__ __forceinline__ bool tight() const {
        const float e = fmaxf(hi.x - lo.x, fmaxf(hi.y - lo.y, hi.z - lo.z));
        return e * e <= 16.0f * r2;
    }
    // The gap between the boxes per axis, max(blo - hi, lo - bhi, 0), then d2
    // as hits() forms it.
    __device__ __forceinline__ bool meets(float3 blo, float3 bhi) const {
        float ax, ay, bx, by;
        unpack2(add2(pack2(blo.x, blo.y), pack2(-hi.x, -hi.y)), ax, ay);
        unpack2(fma2(pack2(bhi.x, bhi.y), pack2(-1.0f, -1.0f), pack2(lo.x, lo.y)), bx, by);
        const float ex = max3(ax, bx, 0.0f), ey = max3(ay, by, 0.0f);
        const float ez = max3(__fsub_rn(blo.z, hi.z), __fsub_rn(lo.z, bhi.z), 0.0f);
        return __fmaf_rn(ez, ez, __fmaf_rn(ey, ey, __fmul_rn(ex, ex))) <= r2;
    }
};

template <>
struct Region<Box> {
    Box u;          // the union of the query boxes
    float3 size;    // the largest extent of one of them
    __device__ __forceinline__ void gather(const Box &q, bool use) {
        const float inf = __int_as_float(0x7f800000);
        u.lo = make_float3(warp_min(use ? q.lo.x : inf), warp_min(use ? q.lo.y : inf), warp_min(use ? q.lo.z : inf));
        u.hi = make_float3(warp_max(use ? q.hi.x : -inf), warp_max(use ? q.hi.y : -inf),
                           warp_max(use ? q.hi.z : -inf));
        size = make_float3(warp_max(use ? q.hi.x - q.lo.x : 0.0f), warp_max(use ? q.hi.y - q.lo.y : 0.0f),
                           warp_max(use ? q.hi.z - q.lo.z : 0.0f));
    }
    static __device__ __forceinline__ bool hopeless(const Box &q) {
        return isnan(q.lo.x) || isnan(q.lo.y) || isnan(q.lo.z) || isnan(q.hi.x) || isnan(q.hi.y) || isnan(q.hi.z);
    }
    __device__ __forceinline__ bool tight() const {
        return u.hi.x - u.lo.x <= 3.0f * size.x && u.hi.y - u.lo.y <= 3.0f * size.y &&
               u.hi.z - u.lo.z <= 3.0f * size.z;
    }
    __device__ __forceinline__ bool meets(float3 blo, float3 bhi) const { return hits(u, blo, bhi); }
    // The axes along which a query is not much smaller than the largest one
    // there (bit 0: x). Rods along x beside rods along y share a region that none
    // of them comes near to filling; those of one shape do not.
    static constexpr bool kShapes = true;
    __device__ __forceinline__ uint32_t shape(const Box &q) const {
        return (8.0f * (q.hi.x - q.lo.x) >= size.x ? 1u : 0u) | (8.0f * (q.hi.y - q.lo.y) >= size.y ? 2u : 0u) |
               (8.0f * (q.hi.z - q.lo.z) >= size.z ? 4u : 0u);
    }
    // Leaf blocks like this one are so small that queries of another shape may pass
    // them by. (Rods among rods: every block is as long as a rod along all axes.)
    __device__ __forceinline__ bool passes(float3 blo, float3 bhi) const {
        return 2.0f * (bhi.x - blo.x) <= size.x && 2.0f * (bhi.y - blo.y) <= size.y && 2.0f * (bhi.z - blo.z) <= size.z;
    }
};

// ---------------------------------------------------------------- packets

constexpr int kPacketWarps = 4;
// CTAs per SM: points at 32 registers and full occupancy (walk of 2^25 uniform
// points 7.64 ms, 8.97 with 12 CTAs at 40 registers), boxes at 40 (2^25 boxes
// 8.30 ms, 8.56 at 32).
template <int kP>
constexpr int kPacketCtas = kP == LBVH_PRIM_POINTS ? 16 : 12;
// Stack of a packet: a step takes four blocks (at most 28 more entries than
// before) up to kStackFour entries and one block beyond, which adds at most
// 7 entries for each of the 8 heights below the root's children and 8 at the
// end: 48 - 4 + 32 + 7 * 8 + 8 = 140 at most.
constexpr int kStack = 144, kStackFour = 48;
constexpr int kLeafList = 256;   // leaf blocks waiting to be read
constexpr int kCand = 64;        // candidate ring: a full set of 32 and the one being filled

// 16-byte alignment: the candidates are read four at a time, and a CTA holds one of these per warp.
template <int kP>
struct alignas(16) PacketSmem {
    static constexpr int kDim = kP == LBVH_PRIM_POINTS ? 3 : 6;
    float cand[kDim][kCand];
    uint32_t id[kCand];
    uint32_t list[kStack + kLeafList];  // the stack, then the leaf blocks
};
static_assert(sizeof(PacketSmem<LBVH_PRIM_POINTS>) % 16 == 0 && sizeof(PacketSmem<LBVH_PRIM_BOXES>) % 16 == 0 &&
                  (kCand * sizeof(float)) % 16 == 0,
              "rows of candidates start on 16-byte boundaries");

// The lane's query against the 32 candidates at `base` of the ring: bit 31 - j
// = hit of candidate j. For a sphere and points, the gap c - clamp(c, p, p) is
// c - p, taken as p - c (the same magnitude, squared), two candidates per
// instruction; the sign of r2 - d2 says d2 > r2 exactly, and it is shifted
// into the mask (an infinite d2 against an infinite r2 gives the canonical
// NaN, whose sign is clear: a hit, as d2 <= r2).
template <int kP>
__device__ __forceinline__ uint32_t test32(const PacketSmem<kP> &sm, int base, const Sphere &q) {
    if constexpr (kP == LBVH_PRIM_POINTS) {
        uint32_t miss = 0;
        const uint64_t nx = pack2(-q.c.x, -q.c.x), ny = pack2(-q.c.y, -q.c.y), nz = pack2(-q.c.z, -q.c.z);
        const uint64_t r2 = pack2(q.r2, q.r2), neg = pack2(-1.0f, -1.0f);
#pragma unroll
        for (int j = 0; j < 32; j += 4) {
            const ulonglong2 x = *reinterpret_cast<const ulonglong2 *>(&sm.cand[0][base + j]);
            const ulonglong2 y = *reinterpret_cast<const ulonglong2 *>(&sm.cand[1][base + j]);
            const ulonglong2 z = *reinterpret_cast<const ulonglong2 *>(&sm.cand[2][base + j]);
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                const uint64_t ex = add2(h ? x.y : x.x, nx), ey = add2(h ? y.y : y.x, ny), ez = add2(h ? z.y : z.x, nz);
                float a, b;
                unpack2(fma2(fma2(ez, ez, fma2(ey, ey, mul2(ex, ex))), neg, r2), a, b);
                miss = __funnelshift_l(__float_as_uint(a), miss, 1);
                miss = __funnelshift_l(__float_as_uint(b), miss, 1);
            }
        }
        return ~miss;
    } else {
        uint32_t mask = 0;
#pragma unroll 8
        for (int j = 0; j < 32; ++j) {
            const float3 lo = make_float3(sm.cand[0][base + j], sm.cand[1][base + j], sm.cand[2][base + j]);
            const float3 hi = make_float3(sm.cand[3][base + j], sm.cand[4][base + j], sm.cand[5][base + j]);
            if (hits(q, lo, hi)) mask |= 0x80000000u >> j;
        }
        return mask;
    }
}

// A box: q.lo <= hi and lo <= q.hi on every axis, as the signs of hi - q.lo
// and q.hi - lo, two candidates per instruction; one sign bit set is a miss.
// Rounding keeps the sign of a difference, and equal values give +0, except
// zeros: (-0) - (+0) is -0. So the query's bounds come in as 0 - q.lo and
// q.hi + 0, which are +0 for either zero (2^24 box queries on 2^25 boxes, build
// and query: 10.73 ms with the bounds as they are, 10.49 with these).
template <int kP>
__device__ __forceinline__ uint32_t test32(const PacketSmem<kP> &sm, int base, const Box &q) {
    constexpr int kHi = kP == LBVH_PRIM_POINTS ? 0 : 3;
    const float minus_lo[3] = {__fsub_rn(0.0f, q.lo.x), __fsub_rn(0.0f, q.lo.y), __fsub_rn(0.0f, q.lo.z)};
    const float plus_hi[3] = {__fadd_rn(q.hi.x, 0.0f), __fadd_rn(q.hi.y, 0.0f), __fadd_rn(q.hi.z, 0.0f)};
    const uint64_t neg = pack2(-1.0f, -1.0f);
    uint32_t miss = 0;
#pragma unroll
    for (int j = 0; j < 32; j += 4) {
        uint32_t s[4] = {0u, 0u, 0u, 0u};
#pragma unroll
        for (int d = 0; d < 3; ++d) {
            const ulonglong2 lo = *reinterpret_cast<const ulonglong2 *>(&sm.cand[d][base + j]);
            const ulonglong2 hi = kHi ? *reinterpret_cast<const ulonglong2 *>(&sm.cand[kHi + d][base + j]) : lo;
            const uint64_t nl = pack2(minus_lo[d], minus_lo[d]), h = pack2(plus_hi[d], plus_hi[d]);
#pragma unroll
            for (int k = 0; k < 2; ++k) {
                float a, b, c, e;
                unpack2(add2(k ? hi.y : hi.x, nl), a, b);
                unpack2(fma2(k ? lo.y : lo.x, neg, h), c, e);
                s[2 * k] |= __float_as_uint(a) | __float_as_uint(c);
                s[2 * k + 1] |= __float_as_uint(b) | __float_as_uint(e);
            }
        }
#pragma unroll
        for (int k = 0; k < 4; ++k) miss = __funnelshift_l(s[k], miss, 1);
    }
    return ~miss;
}

// The packet of the lanes with `use` set walks one tree; k.take(m, sm, ring, q)
// gets every set of candidates with the lane's hits among them (bit 31 - j:
// candidate ring + j). Warp-wide. If more than kLeafList - 32 leaf blocks meet
// its region, a packet that is not tight gives up with nothing taken, and so does a
// whole one (not yet cut) of several shapes if those blocks are small; `shape` is
// then the lane's.
// Keep::kMaxBlocks (0: none): past this many leaf blocks the walk gives up as
// well (k.reset() drops what its own lanes took; the others may hold what an
// earlier packet gave them), and a lane is out once k.full().
enum Walked : int { kWalked, kTooLoose, kUnlike };

template <int kQ, int kP, typename Keep>
__device__ __forceinline__ Walked packet_walk(const Blocks &t, PacketSmem<kP> &sm, const typename QueryOf<kQ>::type &q,
                                              bool use, bool whole, uint32_t &shape, Keep &k) {
    using Q = typename QueryOf<kQ>::type;
    const int lane = threadIdx.x & 31, sub = lane >> 3;
    const uint32_t below = (1u << lane) - 1u;
    Region<Q> region;
    const bool mine = use;
    use = use && !Region<Q>::hopeless(q);
    if (!__any_sync(kFull, use)) return kWalked;
    region.gather(q, use);
    const bool tight = region.tight();
    int ns = 0, nl = 0;      // entries of the stack and of the leaf list
    int ring = 0, nc = 0;    // candidates: the set of 32 being filled starts at `ring`
    bool fresh = true;       // no leaf block has been read yet
    int read = 0;            // leaf blocks read (counted with kMaxBlocks)
    if (lane == 0) sm.list[t.start0 ? 0 : kStack] = 0u;
    if (t.start0) ns = 1;
    else nl = 1;
    __syncwarp();
    // tests the full (or, at the end, last) set of candidates
    auto flush = [&](int count) {
        uint32_t m = test32<kP>(sm, ring, q);
        if (count < 32) m &= ~(kFull >> count);
        if (!use) m = 0;
        k.take(m, sm, ring, q);
    };
    while (true) {
        // ---- blocks: until the leaf list could overflow in the next step
        while (ns > 0 && nl <= kLeafList - 32) {
            const int take = ns > kStackFour ? 1 : min(4, ns);
            ns -= take;
            bool hit = false;
            uint32_t child = 0;
            if (sub < take) {
                child = sm.list[ns + sub] * kFan + 1u + (lane & 7);
                float4 a, b;
                ld_node32(t.rec + 2 * (int64_t)child, a, b);
                hit = region.meets(xyz(a), xyz(b)) && __float_as_uint(b.w) == kBlockExists;
            }
            const bool leaf = child >= t.start0;
            const uint32_t inner = __ballot_sync(kFull, hit && !leaf), leafs = __ballot_sync(kFull, hit && leaf);
            if (hit) sm.list[(leaf ? kStack + nl : ns) + __popc((leaf ? leafs : inner) & below)] = child;
            ns += __popc(inner);
            nl += __popc(leafs);
            __syncwarp();
        }
        if (ns > 0 && fresh) {
            if (!tight) return kTooLoose;
            if constexpr (Region<Q>::kShapes) {
                if (whole) {
                    region.gather(q, use);  // (its sizes were not kept in registers)
                    shape = region.shape(q);
                    const uint32_t one = __shfl_sync(kFull, shape, __ffs(__ballot_sync(kFull, use)) - 1);
                    float4 a, b;
                    ld_node32(t.rec + 2 * (int64_t)sm.list[kStack + lane], a, b);  // one of the leaf blocks
                    const uint32_t small = __ballot_sync(kFull, region.passes(xyz(a), xyz(b)));
                    if (__any_sync(kFull, use && shape != one) && __popc(small) >= 16) return kUnlike;
                }
            }
        }
        fresh = false;
        if constexpr (Keep::kMaxBlocks > 0) {
            read += nl;
            if (read > Keep::kMaxBlocks) {
                if (mine) k.reset();
                return kTooLoose;
            }
        }
        // ---- leaves
        while (nl > 0) {
            const int take = min(4, nl);
            nl -= take;
            bool in = false;
            float4 a = make_float4(0.f, 0.f, 0.f, 0.f), b = a;
            if (sub < take) {
                const int pos = (int)(sm.list[kStack + nl + sub] - t.start0) * kFan + (lane & 7);
                if (pos < t.n) {
                    if (kP == LBVH_PRIM_BOXES) {
                        ld_node32(t.leaves + 2 * (int64_t)pos, a, b);
                    } else {
                        a = __ldg(t.leaves + pos);
                        b = a;
                    }
                    in = region.meets(leaf_lo<kP>(a, b), leaf_hi<kP>(a, b));
                }
            }
            const uint32_t got = __ballot_sync(kFull, in);
            if (in) {
                const int at = (ring + nc + __popc(got & below)) & (kCand - 1);
                sm.cand[0][at] = a.x;
                sm.cand[1][at] = a.y;
                sm.cand[2][at] = a.z;
                if constexpr (kP == LBVH_PRIM_BOXES) {
                    sm.cand[3][at] = b.x;
                    sm.cand[4][at] = b.y;
                    sm.cand[5][at] = b.z;
                }
                sm.id[at] = __float_as_uint(a.w) & kLeafIndexMask;
            }
            nc += __popc(got);
            __syncwarp();
            if (nc >= 32) {
                flush(32);
                ring ^= 32;
                nc -= 32;
                __syncwarp();
                if constexpr (Keep::kMaxBlocks > 0) {
                    const bool out = use && k.full();
                    if (__any_sync(kFull, out)) {  // the region of the others
                        use = use && !out;
                        if (!__any_sync(kFull, use)) return kWalked;
                        region.gather(q, use);
                    }
                }
            }
        }
        if (ns == 0) break;
    }
    if (nc > 0) flush(nc);
    __syncwarp();
    return kWalked;
}

__device__ __forceinline__ float3 middle(const Sphere &s) { return s.c; }
__device__ __forceinline__ float3 middle(const Box &b) {
    return make_float3(b.lo.x + b.hi.x, b.lo.y + b.hi.y, b.lo.z + b.hi.z);
}

// The lanes of `mine` before its widest step from one query to the next (the
// order may be a Morton curve, which jumps now and then, or queries may be
// scarce on their curve: such a packet is two packets far apart). `mine` is a run of lanes, two at least.
template <typename Q>
__device__ __forceinline__ uint32_t before_jump(const Q &q, uint32_t mine) {
    const int lane = threadIdx.x & 31;
    const float3 c = middle(q);
    const float dx = c.x - __shfl_up_sync(kFull, c.x, 1), dy = c.y - __shfl_up_sync(kFull, c.y, 1),
                dz = c.z - __shfl_up_sync(kFull, c.z, 1);
    const float d = fmaxf(fabsf(dx), fmaxf(fabsf(dy), fabsf(dz)));
    const bool step = ((mine >> lane) & 1u) && lane > __ffs(mine) - 1;
    const float widest = warp_max(step && d >= 0.0f ? d : 0.0f);
    const uint32_t at = __ballot_sync(kFull, step && d == widest);
    const int cut = at ? __ffs(at) - 1 : __ffs(mine);
    return mine & ((1u << cut) - 1u);
}

// The queries of `mine` (a run of lanes of one tree): as one packet, or, where
// that gave up, as two on either side of the widest jump, or one for each shape
// (queries on as many points, whole call, as one packet / by shapes: 300,000 rods
// of 0.2 x 0.002^2 along random axes 750 / 305 us, Algorithm 1 256; 10^6 rods
// of half the size 1135 / 525, 448; 2 * 10^6 plates of 0.07^2 x 0.001 2262 / 2252,
// 2771). Returns the lanes left over, whose queries lie too far apart.
template <int kQ, int kP, typename Keep>
__device__ __forceinline__ uint32_t packets(const Blocks &t, PacketSmem<kP> &sm, const typename QueryOf<kQ>::type &q,
                                            uint32_t mine, Keep &k) {
    const int lane = threadIdx.x & 31;
    uint32_t cur = mine, rest = 0, left = 0, shape = 0;
    bool whole = true, by_shape = false;
    while (cur) {
        const Walked w = packet_walk<kQ, kP>(t, sm, q, (cur >> lane) & 1u, whole, shape, k);
        if (w == kUnlike) {
            by_shape = true;
            rest = cur;
        } else if (w == kTooLoose && whole && __popc(cur) > 1) {
            const uint32_t first = before_jump(q, cur);
            rest = cur & ~first;
            cur = first;
            whole = false;
            continue;
        } else if (w == kTooLoose) {
            left |= cur;
        }
        whole = false;
        cur = rest;
        if (by_shape && rest)  // the first lane's shape
            cur &= __ballot_sync(kFull, shape == __shfl_sync(kFull, shape, __ffs(rest) - 1));
        rest &= ~cur;
    }
    return left;
}

}  // namespace lbvh
