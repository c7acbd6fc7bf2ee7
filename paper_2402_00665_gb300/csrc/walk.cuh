// walk.cuh -- what the collecting walks share (query.cu: Algorithm 1 over the
// tree's nodes; packet.cu: packets of queries over the boxes of leaf blocks):
// the query types and their predicates, the node load, and the query scratch.
#pragma once

#include "lbvh_internal.cuh"

namespace lbvh {

// f32x2: two FP32 operations of one instruction, each rounded as its scalar form
__device__ __forceinline__ uint64_t pack2(float a, float b) {
    uint64_t r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(a), "f"(b));
    return r;
}
__device__ __forceinline__ void unpack2(uint64_t v, float &a, float &b) {
    asm("mov.b64 {%0, %1}, %2;" : "=f"(a), "=f"(b) : "l"(v));
}
__device__ __forceinline__ uint64_t add2(uint64_t a, uint64_t b) {
    uint64_t r;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}
__device__ __forceinline__ uint64_t mul2(uint64_t a, uint64_t b) {
    uint64_t r;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}
__device__ __forceinline__ uint64_t fma2(uint64_t a, uint64_t b, uint64_t c) {
    uint64_t r;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
    return r;
}

__device__ __forceinline__ float max3(float a, float b, float c) {
    float r;
    asm("max.f32 %0, %1, %2, %3;" : "=f"(r) : "f"(a), "f"(b), "f"(c));
    return r;
}
__device__ __forceinline__ float min3(float a, float b, float c) {
    float r;
    asm("min.f32 %0, %1, %2, %3;" : "=f"(r) : "f"(a), "f"(b), "f"(c));
    return r;
}

struct Sphere {
    float3 c;
    float r2;
};
struct Box {
    float3 lo, hi;
};
// A ray segment: origin, 1/direction per axis (IEEE division), which axes
// are parallel (direction 0, or a reciprocal that overflows), and [tmin, tmax].
struct Ray {
    float3 o, inv;
    float tmin, tmax;
    uint32_t parallel;  // bit a: axis a
};

// |gap| between c and [lo, hi]: c - clamp(c, lo, hi) (sign irrelevant: squared)
__device__ __forceinline__ float gap(float lo, float c, float hi) {
    return __fsub_rn(c, fminf(fmaxf(c, lo), hi));
}

// Squared distance from c to the box: ex*ex, then + ey*ey and + ez*ez each
// as one fused multiply-add.
__device__ __forceinline__ float box_d2(float3 c, float3 lo, float3 hi) {
    const float ex = gap(lo.x, c.x, hi.x);
    const float ey = gap(lo.y, c.y, hi.y);
    const float ez = gap(lo.z, c.z, hi.z);
    return __fmaf_rn(ez, ez, __fmaf_rn(ey, ey, __fmul_rn(ex, ex)));
}

__device__ __forceinline__ bool hits(const Sphere &s, float3 lo, float3 hi) { return box_d2(s.c, lo, hi) <= s.r2; }

// Slab test, each operation rounded once: per axis t1 = (lo - o) * inv and
// t2 = (hi - o) * inv; tnear = max(tmin, min(t1, t2)), tfar = min(tmax,
// max(t1, t2)); a parallel axis instead requires lo <= o <= hi. Hit iff
// tnear <= tfar. Monotone in the box, like the other predicates.
__device__ __forceinline__ bool slab(float lo, float hi, float o, float inv, bool parallel, float &tn,
                                     float &tf) {
    if (parallel) return lo <= o && o <= hi;
    const float t1 = __fmul_rn(__fsub_rn(lo, o), inv), t2 = __fmul_rn(__fsub_rn(hi, o), inv);
    tn = fmaxf(tn, fminf(t1, t2));
    tf = fminf(tf, fmaxf(t1, t2));
    return true;
}

__device__ __forceinline__ bool hits(const Ray &r, float3 lo, float3 hi) {
    float tn = r.tmin, tf = r.tmax;
    if (!slab(lo.x, hi.x, r.o.x, r.inv.x, r.parallel & 1u, tn, tf)) return false;
    if (!slab(lo.y, hi.y, r.o.y, r.inv.y, r.parallel & 2u, tn, tf)) return false;
    if (!slab(lo.z, hi.z, r.o.z, r.inv.z, r.parallel & 4u, tn, tf)) return false;
    return tn <= tf;
}

// A ray without a parallel axis: the same operations on every axis, x and y
// in one instruction each and the extremes three at a time (they do not
// depend on the order; no operand is NaN).
struct SlantedRay : Ray {};
__device__ __forceinline__ bool hits(const SlantedRay &r, float3 lo, float3 hi) {
    const uint64_t minus = pack2(-r.o.x, -r.o.y), inv = pack2(r.inv.x, r.inv.y);
    float ax, ay, bx, by;
    unpack2(mul2(add2(pack2(lo.x, lo.y), minus), inv), ax, ay);
    unpack2(mul2(add2(pack2(hi.x, hi.y), minus), inv), bx, by);
    const float az = __fmul_rn(__fsub_rn(lo.z, r.o.z), r.inv.z), bz = __fmul_rn(__fsub_rn(hi.z, r.o.z), r.inv.z);
    const float tn = max3(max3(fminf(ax, bx), fminf(ay, by), fminf(az, bz)), r.tmin, r.tmin);
    const float tf = min3(min3(fmaxf(ax, bx), fmaxf(ay, by), fmaxf(az, bz)), r.tmax, r.tmax);
    return tn <= tf;
}

__device__ __forceinline__ bool hits(const Box &q, float3 lo, float3 hi) {
    return q.lo.x <= hi.x && lo.x <= q.hi.x && q.lo.y <= hi.y && lo.y <= q.hi.y &&
           q.lo.z <= hi.z && lo.z <= q.hi.z;
}

template <int kQ>
struct QueryOf;
template <>
struct QueryOf<LBVH_Q_SPHERE> {
    using type = Sphere;
    static __device__ __forceinline__ Sphere load(const QueryArgs &a, int64_t q) {
        const float *p = a.queries + 3 * q;
        const float r = a.radii ? __ldcs(a.radii + q) : a.radius;
        return Sphere{make_float3(__ldcs(p), __ldcs(p + 1), __ldcs(p + 2)), __fmul_rn(r, r)};
    }
};
template <>
struct QueryOf<LBVH_Q_RAY> {
    using type = Ray;
    static __device__ __forceinline__ float axis_inv(float d, uint32_t bit, uint32_t &parallel) {
        const float inv = __fdiv_rn(1.0f, d);
        if (d == 0.0f || isinf(inv)) parallel |= bit;
        return inv;
    }
    static __device__ __forceinline__ Ray load(const QueryArgs &a, int64_t q) {
        const float4 *p = reinterpret_cast<const float4 *>(a.queries) + 2 * q;
        const float4 u = __ldcs(p), v = __ldcs(p + 1);
        Ray r;
        r.parallel = 0;
        r.o = make_float3(u.x, u.y, u.z);
        r.inv = make_float3(axis_inv(v.x, 1u, r.parallel), axis_inv(v.y, 2u, r.parallel),
                            axis_inv(v.z, 4u, r.parallel));
        r.tmin = u.w;
        r.tmax = v.w;
        const bool finite = isfinite(u.x) && isfinite(u.y) && isfinite(u.z) && isfinite(v.x) && isfinite(v.y) &&
                            isfinite(v.z) && !isnan(u.w) && !isnan(v.w);
        if (!finite) {  // hits nothing: an empty parameter interval on every axis
            r.tmin = 1.0f;
            r.tmax = 0.0f;
            r.parallel = 0;
            r.o = make_float3(0.0f, 0.0f, 0.0f);
            r.inv = make_float3(1.0f, 1.0f, 1.0f);
        }
        return r;
    }
};
template <>
struct QueryOf<LBVH_Q_BOX> {
    using type = Box;
    static __device__ __forceinline__ Box load(const QueryArgs &a, int64_t q) {
        const float *p = a.queries + 6 * q;
        return Box{make_float3(__ldcs(p), __ldcs(p + 1), __ldcs(p + 2)),
                   make_float3(__ldcs(p + 3), __ldcs(p + 4), __ldcs(p + 5))};
    }
};

__device__ __forceinline__ float3 xyz(float4 v) { return make_float3(v.x, v.y, v.z); }

// A node record as one 32-byte load (two float4 halves), read-only path.
// Records of two float4 start on 32-byte boundaries (internal nodes and box
// leaves; batches pad every tree to an even float4 offset).
__device__ __forceinline__ void ld_node32(const float4 *p, float4 &a, float4 &b) {
    asm("ld.global.nc.v8.f32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
        : "=f"(a.x), "=f"(a.y), "=f"(a.z), "=f"(a.w), "=f"(b.x), "=f"(b.y), "=f"(b.z), "=f"(b.w)
        : "l"(p));
}

// The node at `unit` (float4 units). In a box tree every record is 32 bytes:
// one 32-byte load per step (measured: D3's walk 10.14 -> 8.39 ms). In a
// point tree a leaf is one float4 (its box is its point): a first 16-byte
// load common to every lane and a second one for internal nodes measured
// faster than splitting the warp between a 16- and a 32-byte load.
template <int kP>
__device__ __forceinline__ void load_node(const float4 *base, int unit, bool leaf, float4 &a, float4 &b) {
    if (kP == LBVH_PRIM_BOXES) {
        ld_node32(base + unit, a, b);
    } else {
        a = __ldg(base + unit);
        b = a;
        if (!leaf) b = __ldg(base + unit + 1);
    }
}

constexpr int kSlot = kQueryBufferHits;  // ids kept per walk (slot size)
constexpr int kRegSort = 32;             // lists up to this long are sorted in one thread's registers

// The query of walk position i. The order of a sort that gave up a wait holds
// words it never wrote: whatever they are, no query past the last is indexed.
__device__ __forceinline__ int64_t thread_query(const QueryArgs &qa, int64_t i) {
    return qa.order ? min((int64_t)__ldcs(qa.order + i), qa.nq - 1) : i;
}
// The same where the queries may be rays, whose order is not always used.
template <int kQ>
__device__ __forceinline__ int64_t query_at(const QueryArgs &qa, int64_t i) {
    if (kQ == LBVH_Q_RAY && qa.apart && *qa.apart < qa.apart_min) return i;
    return thread_query(qa, i);
}

// Hits past a walk's slot: appended to chunks from the shared pool, the first
// chunk recorded in spill_head[q], each chunk's word 0 linking to the next.
// `cur` is the walk's current chunk (kNoChunk before the first); it becomes
// kSpillFailed when the pool is exhausted, and the query then takes the
// second walk.
constexpr uint32_t kNoChunk = 0xffffffffu, kSpillFailed = 0xfffffffeu;

__device__ __forceinline__ void spill_put(const QueryScratch &qs, Control *ctl, int64_t i, uint32_t cnt,
                                          uint32_t id, uint32_t &cur) {
    if (cur == kSpillFailed) return;
    const uint32_t sidx = cnt - (uint32_t)kSlot;                   // index among the spilled hits
    const uint32_t off = sidx % (uint32_t)(kSpillChunkWords - 1);  // slot in the chunk (after the link)
    if (off == 0) {
        const uint32_t fresh = atomicAdd(&ctl->spill_used, 1u);
        if (fresh >= qs.spill_chunks) {
            cur = kSpillFailed;
            return;
        }
        if (cur == kNoChunk) qs.spill_head[i] = fresh;
        else qs.spill[(int64_t)cur * kSpillChunkWords] = fresh;
        cur = fresh;
    }
    qs.spill[(int64_t)cur * kSpillChunkWords + 1 + off] = id;
}

// ---------------------------------------------------------------- leaf blocks (packet.cu)

constexpr uint32_t kFull = 0xffffffffu;
constexpr int kFan = 8;  // children per block
constexpr uint32_t kBlockExists = 1u;

// One tree's blocks as a walk sees them: the leaves, the records, the first
// record of the leaf blocks.
struct Blocks {
    const float4 *leaves, *rec;
    int n;
    uint32_t start0;
};

// The walk of one query by 8 lanes: the lanes test the 8 children of one block
// at a time with the query's own predicate; `stack`: kSparseStack words of
// shared memory per 8 lanes. Warp-wide; `go`: the 8 lanes have a query (qi).
constexpr int kSparseStack = 80;  // one block per step: 7 entries per height (9 below the root) and 8 at the end

template <int kP, typename Q>
__device__ __forceinline__ void sparse_walk(const Blocks &t, uint32_t *stack, const Q &q, bool go, int64_t qi, const QueryScratch &qs,
                                            Control *ctl) {
    const int lane = threadIdx.x & 31, sl = lane & 7, shift = lane & 24;
    const uint32_t below = (1u << sl) - 1u;
    uint32_t *slot = qs.slots + qi * kSlot;
    uint32_t cnt = 0, cur = kNoChunk;
    int ns = 0;
    if (go) {
        if (sl == 0) stack[0] = 0u;
        ns = 1;
    }
    __syncwarp();
    while (__any_sync(kFull, ns > 0)) {
        const bool act = ns > 0;
        const uint32_t item = act ? stack[ns - 1] : 0u;
        const bool leaf = item >= t.start0;  // a leaf block: its children are leaves
        const uint32_t child = (leaf ? (item - t.start0) * kFan : item * kFan + 1u) + sl;
        bool hit = false;
        uint32_t id = 0;
        if (act && !(leaf && child >= (uint32_t)t.n)) {
            float4 a, b;
            if (kP == LBVH_PRIM_BOXES) {
                ld_node32((leaf ? t.leaves : t.rec) + 2 * (int64_t)child, a, b);
            } else {
                const float4 *p = leaf ? t.leaves + child : t.rec + 2 * (int64_t)child;
                a = __ldg(p);
                b = a;
                if (!leaf) b = __ldg(p + 1);
            }
            hit = hits(q, xyz(a), xyz(b)) && (leaf || __float_as_uint(b.w) == kBlockExists);
            id = __float_as_uint(a.w) & kLeafIndexMask;
        }
        const uint32_t bits = (__ballot_sync(kFull, hit) >> shift) & 0xffu;
        if (act) --ns;
        __syncwarp();  // every lane has read its item
        if (!leaf) {
            if (hit) stack[ns + __popc(bits & below)] = child;
            ns += __popc(bits);
        } else if (bits) {
            const uint32_t at = cnt + __popc(bits & below), m = (uint32_t)__popc(bits);
            if (hit && at < (uint32_t)kSlot) __stcs(slot + at, id);
            if (cnt + m > (uint32_t)kSlot) {  // past the slot: in order, one lane after the other
                const uint32_t mates = 0xffu << shift;
                for (uint32_t r = bits; r; r &= r - 1) {
                    const int src = shift + __ffs(r) - 1;
                    const uint32_t a = __shfl_sync(mates, at, src), v = __shfl_sync(mates, id, src);
                    if (a >= (uint32_t)kSlot && sl == 0) spill_put(qs, ctl, qi, a, v, cur);
                }
            }
            cnt += m;
        }
        __syncwarp();
    }
    if (go && sl == 0) {
        __stcs(qs.counts + qi, cnt);
        if (cnt > (uint32_t)kSlot)
            qs.overflow_list[atomicAdd(&ctl->overflow_filled, 1u)] =
                (uint32_t)qi | (cur != kSpillFailed ? kSpilledTag : 0u);
    }
}

}  // namespace lbvh
