// morton.cuh -- the Morton code of a centroid (Sec. 3.1, Karras step 1), as
// device functions shared by the encoder and by the construct, which derives
// each leaf's code again from the primitive it gathers. Both must compute the
// same bits, so both call these functions.
//
// The paper leaves the encoding open. The one used here:
//   centroid    a point itself; a box (lo + hi) * 0.5 in FP32
//   quantise    t = (c - min) / (max - min), IEEE FP32 subtract and divide;
//               v = t * 2^b (exact); cell = 0 if !(v > 0), 2^b - 1 if
//               v >= 2^b - 1, else trunc(v); cell = 0 on an axis of zero extent
//   interleave  bit 3k+2 = x_k, 3k+1 = y_k, 3k = z_k
// Every float operation is an explicit round-to-nearest intrinsic so the
// compiler cannot contract or reassociate them.
#pragma once

#include <cfloat>
#include <cstdint>

#include "lbvh_internal.cuh"

namespace lbvh {

// Mask of the bit positions that input bit k occupies after the spreading
// steps of levels >= L: bit k has moved up by 2 * (k with its low L bits
// cleared). At level 0 every bit k sits at 3k.
constexpr uint64_t spread_mask(int level) {
    uint64_t m = 0;
    for (int k = 0; k < 21; ++k) m |= 1ull << (k + 2 * (k & ~((1 << level) - 1)));
    return m;
}

// Moves bit k of a 21-bit value to bit 3k.
__device__ __forceinline__ uint64_t spread3(uint32_t v) {
    uint64_t x = v & 0x1fffffu;
    x = (x | (x << 32)) & spread_mask(4);
    x = (x | (x << 16)) & spread_mask(3);
    x = (x | (x << 8)) & spread_mask(2);
    x = (x | (x << 4)) & spread_mask(1);
    x = (x | (x << 2)) & spread_mask(0);
    return x;
}

// The quantisation grid: scene bounds and 2^b cells per axis.
struct Grid3 {
    float lo[3];
    float extent[3];
    float cells;  // 2^b
    float top;    // 2^b - 1
    uint32_t topi;
};

// bounds: float[6] {min.xyz, max.xyz}; b = code bits / 3.
__device__ __forceinline__ Grid3 make_grid(const float *bounds, int b) {
    Grid3 g;
    for (int a = 0; a < 3; ++a) {
        g.lo[a] = bounds[a];
        g.extent[a] = __fsub_rn(bounds[3 + a], bounds[a]);
    }
    g.topi = (1u << b) - 1u;
    g.cells = (float)(1u << b);
    g.top = (float)g.topi;
    return g;
}

__device__ __forceinline__ uint32_t cell_of(float c, float lo, float extent, const Grid3 &g) {
    if (!(extent > 0.0f)) return 0u;
    const float t = __fdiv_rn(__fsub_rn(c, lo), extent);
    const float v = __fmul_rn(t, g.cells);
    if (!(v > 0.0f)) return 0u;
    if (v >= g.top) return g.topi;
    return __float2uint_rz(v);
}

__device__ __forceinline__ uint64_t morton(float x, float y, float z, const Grid3 &g) {
    const uint32_t qx = cell_of(x, g.lo[0], g.extent[0], g);
    const uint32_t qy = cell_of(y, g.lo[1], g.extent[1], g);
    const uint32_t qz = cell_of(z, g.lo[2], g.extent[2], g);
    return (spread3(qx) << 2) | (spread3(qy) << 1) | spread3(qz);
}

// ---- Hilbert order (queries only: neighbours on the curve are neighbours in
// space, without the Morton curve's jumps; the order of the queries changes
// no result). One level at a time with the entry point e and direction d of
// the cell (C. Hamilton, "Compact Hilbert Indices", 2006): the octant l
// becomes t = rotr(l ^ e, d + 1), its rank on the curve is the inverse Gray
// code w of t, and the child's e ^= rotl(entry(w), d + 1), d += dir(w) + 1.
// The table takes two levels at once: for state e * 3 + d and the 6 bits of
// two octants, their 6 bits on the curve | next state << 6.
constexpr int kHilbertStates = 24;
constexpr int kHilbertEntries = kHilbertStates * 64;
struct HilbertTable {
    uint16_t next[kHilbertEntries];
};
constexpr uint32_t rot3(uint32_t v, uint32_t left) {
    left %= 3u;
    return ((v << left) | (v >> (3u - left))) & 7u;
}
constexpr HilbertTable hilbert_table() {
    uint32_t one[kHilbertStates * 8]{};  // one level: 3 bits | next state << 3
    for (uint32_t e = 0; e < 8; ++e)
        for (uint32_t d = 0; d < 3; ++d)
            for (uint32_t l = 0; l < 8; ++l) {
                const uint32_t g = rot3(l ^ e, 3u - (d + 1u) % 3u);
                const uint32_t w = g ^ (g >> 1) ^ (g >> 2);
                const uint32_t before = w == 0 ? 0u : 2u * ((w - 1u) / 2u);  // entry(w) = gray(before)
                const uint32_t ne = e ^ rot3(before ^ (before >> 1), d + 1u);
                // dir(w): trailing ones of w (odd w) or of w - 1 (even w > 0), mod 3
                uint32_t v = w == 0 ? 0u : (w & 1u ? w : w - 1u), dir = 0;
                while (v & 1u) {
                    ++dir;
                    v >>= 1;
                }
                const uint32_t nd = (d + dir + 1u) % 3u;
                one[(e * 3u + d) * 8u + l] = w | (ne * 3u + nd) << 3;
            }
    HilbertTable t{};
    for (uint32_t k = 0; k < (uint32_t)kHilbertEntries; ++k) {
        const uint32_t a = one[(k >> 6) * 8u + ((k >> 3) & 7u)], b = one[(a >> 3) * 8u + (k & 7u)];
        t.next[k] = (uint16_t)((a & 7u) << 3 | (b & 7u) | (b >> 3) << 6);
    }
    return t;
}

// The Hilbert index of a cell of the grid (b bits per axis, at most 21);
// `table`: hilbert_table().next. An odd b is made even by a level
// above, all of it octant 0: state 2 (e = 0, d = 2) takes octant 0 to rank 0
// and state 0. Two levels per step and the octants from the Morton code: the
// order of 2^25 queries 1.305 -> 1.266 ms.
__device__ __forceinline__ uint64_t hilbert(float x, float y, float z, const Grid3 &g, int b, const uint16_t *table) {
    const uint64_t m = morton(x, y, z, g);
    uint64_t code = 0;
    uint32_t state = b & 1 ? 2u << 6 : 0u;
    for (int k = 3 * (b + (b & 1)) - 6; k >= 0; k -= 6) {
        const uint32_t e = table[state | ((uint32_t)(m >> k) & 63u)];
        code = code << 6 | (e & 63u);
        state = e & ~63u;
    }
    return code;
}

__device__ __forceinline__ bool finite3(float x, float y, float z) {
    return fabsf(x) <= FLT_MAX && fabsf(y) <= FLT_MAX && fabsf(z) <= FLT_MAX;
}

__device__ __forceinline__ void box_centroid(const float *b, float &x, float &y, float &z) {
    x = __fmul_rn(__fadd_rn(b[0], b[3]), 0.5f);
    y = __fmul_rn(__fadd_rn(b[1], b[4]), 0.5f);
    z = __fmul_rn(__fadd_rn(b[2], b[5]), 0.5f);
}

// Extremes of finite centroids (min_ordered / max_ordered: lbvh_internal.cuh).
struct MinMax {
    float lo[3], hi[3];
    bool ok;
    __device__ void init() {
        for (int a = 0; a < 3; ++a) {
            lo[a] = FLT_MAX;
            hi[a] = -FLT_MAX;
        }
        ok = true;
    }
    __device__ __forceinline__ void add(float x, float y, float z) {
        ok = ok && finite3(x, y, z);
        lo[0] = min_ordered(lo[0], x);
        lo[1] = min_ordered(lo[1], y);
        lo[2] = min_ordered(lo[2], z);
        hi[0] = max_ordered(hi[0], x);
        hi[1] = max_ordered(hi[1], y);
        hi[2] = max_ordered(hi[2], z);
    }
};

}  // namespace lbvh
