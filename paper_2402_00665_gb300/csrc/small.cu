// small.cu -- scene bounds, Morton codes and their stable sort (Sec. 3.1 steps 1
// and 2) for a small tree, by one CTA in one launch.
//
// A small build is bound by its launches: at 1,000 points the bounds, the
// encoder, four sort passes and two memsets took 68 us, nearly all of it the
// way from one kernel to the next. Here the keys stay in one CTA's shared
// memory. Up to kSmallSort primitives: the keys (8 bytes, and 2 for the index
// beside codes wider than 30 bits) and the warps' digit counts fill 177 KB.
#include "lbvh_internal.cuh"
#include "morton.cuh"
#include "once_per_device.cuh"

namespace lbvh {

namespace {

template <int kKind>
__device__ __forceinline__ void centroid(const float *prims, int i, float &x, float &y, float &z) {
    if (kKind == LBVH_PRIM_POINTS) {
        x = prims[3 * i];
        y = prims[3 * i + 1];
        z = prims[3 * i + 2];
    } else {
        box_centroid(prims + 6 * i, x, y, z);
    }
}

// kWide: codes of more than 30 bits, the index beside the key; else the word
// code << 16 | index. kT threads hold kR keys each.
template <bool kWide, int kT, int kR>
struct SmallSmem {
    uint64_t key[kT * kR];
    uint16_t index[kWide ? kT * kR : 1];
    alignas(16) uint16_t count[kT / 32][kRadix];  // (cleared as 32-bit words) digits of a warp's keys, then of the warps before it in its group of 8
    uint32_t group[kT / 256][kRadix];  // digits of a group of 8 warps, then its first place per digit
    uint32_t warp_sum[kRadix / 32];
    float extreme[kT / 32][6];
    float bounds[6];
    int finite;
};
template <int kKind, bool kWide, int kT, int kR>
__global__ void __launch_bounds__(kT, 1)
    small_sort_kernel(const float *__restrict__ prims, int n, int bits, float *__restrict__ bounds,
                      uint32_t *__restrict__ perm, uint32_t *flags) {
    extern __shared__ __align__(16) unsigned char raw[];
    auto &sm = *reinterpret_cast<SmallSmem<kWide, kT, kR> *>(raw);
    const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
    // ---- scene bounds
    if (t == 0) sm.finite = 1;
    MinMax m;
    m.init();
    for (int i = t; i < n; i += kT) {
        float x, y, z;
        centroid<kKind>(prims, i, x, y, z);
        m.add(x, y, z);
    }
    for (int off = 16; off > 0; off >>= 1)
        for (int a = 0; a < 3; ++a) {
            m.lo[a] = min_ordered(m.lo[a], __shfl_xor_sync(0xffffffffu, m.lo[a], off));
            m.hi[a] = max_ordered(m.hi[a], __shfl_xor_sync(0xffffffffu, m.hi[a], off));
        }
    if (lane < 6) sm.extreme[warp][lane] = lane == 0 ? m.lo[0] : lane == 1 ? m.lo[1] : lane == 2 ? m.lo[2]
                                         : lane == 3 ? m.hi[0] : lane == 4 ? m.hi[1] : m.hi[2];
    __syncthreads();
    if (!m.ok) sm.finite = 0;
    if (t < 6) {
        float v = sm.extreme[0][t];
        for (int w = 1; w < kT / 32; ++w)
            v = t < 3 ? min_ordered(v, sm.extreme[w][t]) : max_ordered(v, sm.extreme[w][t]);
        sm.bounds[t] = v;
        bounds[t] = v;
    }
    __syncthreads();
    if (t == 0 && !sm.finite) atomicOr(flags, kFlagNonfinite);
    // ---- codes (places past n sort last)
    const Grid3 g = make_grid(sm.bounds, bits / 3);
    for (int i = t; i < kT * kR; i += kT) {
        uint64_t k = ~0ull;
        if (i < n) {
            float x, y, z;
            centroid<kKind>(prims, i, x, y, z);
            k = morton(x, y, z, g);
            if (!kWide) k = k << 16 | (uint64_t)i;
        }
        sm.key[i] = k;
        if (kWide) sm.index[i] = (uint16_t)i;
    }
    __syncthreads();
    // ---- LSD passes over 8-bit digits; warp w holds keys [w * 32 kR, (w + 1) * 32 kR), round j lane l key 32 j + l
    const uint32_t below = (1u << lane) - 1u;
    for (int shift = kWide ? 0 : 16; shift < (kWide ? bits : 16 + bits); shift += kRadixBits) {
        uint64_t key[kR];
        uint32_t at[kR];  // index (low half) and rank among the warp's keys of its digit
        for (int d = lane; d < kRadix / 2; d += 32) reinterpret_cast<uint32_t *>(sm.count[warp])[d] = 0;
        __syncwarp();
#pragma unroll
        for (int j = 0; j < kR; ++j) {
            const int e = (warp * kR + j) * 32 + lane;
            key[j] = sm.key[e];
            at[j] = kWide ? sm.index[e] : 0u;
        }
#pragma unroll
        for (int j = 0; j < kR; ++j) {
            const uint32_t d = (uint32_t)(key[j] >> shift) & (kRadix - 1);
            uint32_t peers = 0xffffffffu;
#pragma unroll
            for (int b = 0; b < kRadixBits; ++b) {
                const uint32_t vote = __ballot_sync(0xffffffffu, (d >> b) & 1u);
                peers &= ((d >> b) & 1u) ? vote : ~vote;
            }
            const uint32_t before = __popc(peers & below), base = sm.count[warp][d];
            __syncwarp();
            if (before == 0) sm.count[warp][d] = (uint16_t)(base + __popc(peers));
            __syncwarp();
            at[j] |= (base + before) << 16;
        }
        __syncthreads();
        {
            const int d = t & (kRadix - 1), q = t / kRadix;  // a thread per digit and group of 8 warps
            uint32_t sum = 0;
#pragma unroll
            for (int w = 0; w < 8; ++w) {
                const uint32_t c = sm.count[8 * q + w][d];
                sm.count[8 * q + w][d] = (uint16_t)sum;
                sum += c;
            }
            sm.group[q][d] = sum;
        }
        __syncthreads();
        uint32_t total = 0, incl = 0;
        if (t < kRadix) {
            for (int q = 0; q < kT / 256; ++q) total += sm.group[q][t];
            incl = total;
            for (int off = 1; off < 32; off <<= 1) {
                const uint32_t y = __shfl_up_sync(0xffffffffu, incl, off);
                if (lane >= off) incl += y;
            }
            if (lane == 31) sm.warp_sum[warp] = incl;
        }
        __syncthreads();
        if (t < kRadix) {
            uint32_t first = incl - total;
            for (int w = 0; w < warp; ++w) first += sm.warp_sum[w];
            for (int q = 0; q < kT / 256; ++q) {
                const uint32_t c = sm.group[q][t];
                sm.group[q][t] = first;
                first += c;
            }
        }
        __syncthreads();
#pragma unroll
        for (int j = 0; j < kR; ++j) {
            const uint32_t d = (uint32_t)(key[j] >> shift) & (kRadix - 1);
            const uint32_t to = sm.group[warp >> 3][d] + sm.count[warp][d] + (at[j] >> 16);
            sm.key[to] = key[j];
            if (kWide) sm.index[to] = (uint16_t)at[j];
        }
        __syncthreads();
    }
    for (int i = t; i < n; i += kT) perm[i] = kWide ? (uint32_t)sm.index[i] : (uint32_t)sm.key[i] & 0xffffu;
}

using Kernel = void (*)(const float *, int, int, float *, uint32_t *, uint32_t *);

template <int kKind, bool kWide, int kT, int kR>
void launch(const float *prims, int n, int bits, float *bounds, uint32_t *perm, uint32_t *flags, cudaStream_t s) {
    Kernel k = small_sort_kernel<kKind, kWide, kT, kR>;
    constexpr size_t smem = sizeof(SmallSmem<kWide, kT, kR>);
    static OncePerDevice configured;
    int dev = 0;
    // a failure stays the thread's last error, which the caller's launch check reports
    if (cudaGetDevice(&dev) != cudaSuccess || !configured(dev, [k] {
            return cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem) == cudaSuccess;
        }))
        return;
    k<<<1, kT, smem, s>>>(prims, n, bits, bounds, perm, flags);
}

template <int kKind, bool kWide>
void pick(const float *prims, int n, int bits, float *bounds, uint32_t *perm, uint32_t *flags, cudaStream_t s) {
    if (n <= 1024) launch<kKind, kWide, 256, 4>(prims, n, bits, bounds, perm, flags, s);
    else if (n <= 4096) launch<kKind, kWide, 1024, 4>(prims, n, bits, bounds, perm, flags, s);
    else if (n <= 8192) launch<kKind, kWide, 1024, 8>(prims, n, bits, bounds, perm, flags, s);
    else launch<kKind, kWide, 1024, 16>(prims, n, bits, bounds, perm, flags, s);
}

}  // namespace

void launch_small_sort(const float *prims, int64_t n, int kind, int bits, float *bounds, uint32_t *perm, Control *ctl,
                       cudaStream_t s) {
    static_assert(kSmallSort == 1024 * 16 && kSmallSort <= 1 << 16, "the widest CTA's keys; 16-bit indices");
    const bool wide = bits > 30;
    uint32_t *flags = &ctl->build_flags;
    if (kind == LBVH_PRIM_POINTS)
        (wide ? pick<LBVH_PRIM_POINTS, true> : pick<LBVH_PRIM_POINTS, false>)(prims, (int)n, bits, bounds, perm, flags, s);
    else
        (wide ? pick<LBVH_PRIM_BOXES, true> : pick<LBVH_PRIM_BOXES, false>)(prims, (int)n, bits, bounds, perm, flags, s);
    count_launches(1);
}

}  // namespace lbvh
