// morton.cu -- scene bounds and Morton codes (Sec. 3.1, Karras step 1). The
// encoding itself (centroid, quantisation, interleave) is in morton.cuh.
//
// Both kernels stream the primitives once. Points are read as float4 (three
// float4 = four points per thread step) when the array is 16-byte aligned.
// The encoder also accumulates the global digit histograms of every radix-sort
// pass (shared-memory counters, flushed once per block), which saves the sort
// a separate read of the codes.
#include <cfloat>

#include "lbvh_internal.cuh"
#include "morton.cuh"

namespace lbvh {

namespace {

constexpr int kThreads = 256;

// Visits the centroid of every primitive: f(i, x, y, z). Points go through
// float4 loads when `prims` is 16-byte aligned (4 points per step).
template <int kKind, typename F>
__device__ __forceinline__ void for_each_centroid(const float *prims, int64_t n, F &&f) {
    const int64_t tid = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    if (kKind == LBVH_PRIM_POINTS) {
        const bool vec = (reinterpret_cast<uintptr_t>(prims) & 15u) == 0;
        int64_t head = 0;
        if (vec) {
            const float4 *p4 = reinterpret_cast<const float4 *>(prims);
            const int64_t groups = n / 4;
            for (int64_t g = tid; g < groups; g += stride) {
                const float4 a = p4[3 * g], b = p4[3 * g + 1], c = p4[3 * g + 2];
                f(4 * g + 0, a.x, a.y, a.z);
                f(4 * g + 1, a.w, b.x, b.y);
                f(4 * g + 2, b.z, b.w, c.x);
                f(4 * g + 3, c.y, c.z, c.w);
            }
            head = groups * 4;
        }
        for (int64_t i = head + tid; i < n; i += stride)
            f(i, prims[3 * i], prims[3 * i + 1], prims[3 * i + 2]);
    } else {
        for (int64_t i = tid; i < n; i += stride) {
            float x, y, z;
            box_centroid(prims + 6 * i, x, y, z);
            f(i, x, y, z);
        }
    }
}

template <int kKind>
__global__ void __launch_bounds__(kThreads)
    bounds_kernel(const float *__restrict__ prims, int64_t n, float *__restrict__ partials,
                  float *__restrict__ bounds, Control *__restrict__ ctl) {
    MinMax m;
    m.init();
    for_each_centroid<kKind>(prims, n, [&](int64_t, float x, float y, float z) { m.add(x, y, z); });

    // warp, then block reduction of 6 extrema and the finite flag
    __shared__ float s_v[kThreads / 32][6];
    __shared__ int s_ok[kThreads / 32];
    __shared__ bool s_last;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    int ok = m.ok;
    for (int off = 16; off > 0; off >>= 1) {
        for (int a = 0; a < 3; ++a) {
            m.lo[a] = min_ordered(m.lo[a], __shfl_xor_sync(0xffffffffu, m.lo[a], off));
            m.hi[a] = max_ordered(m.hi[a], __shfl_xor_sync(0xffffffffu, m.hi[a], off));
        }
        ok &= __shfl_xor_sync(0xffffffffu, ok, off);
    }
    if (lane == 0) {
        for (int a = 0; a < 3; ++a) {
            s_v[warp][a] = m.lo[a];
            s_v[warp][3 + a] = m.hi[a];
        }
        s_ok[warp] = ok;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        float v[6];
        int all = 1;
        for (int k = 0; k < 6; ++k) v[k] = s_v[0][k];
        for (int w = 0; w < kThreads / 32; ++w) {
            for (int a = 0; a < 3; ++a) {
                v[a] = min_ordered(v[a], s_v[w][a]);
                v[3 + a] = max_ordered(v[3 + a], s_v[w][3 + a]);
            }
            all &= s_ok[w];
        }
        float *out = partials + 8 * (int64_t)blockIdx.x;
        for (int k = 0; k < 6; ++k) out[k] = v[k];
        out[6] = all ? 1.0f : 0.0f;
        __threadfence();
        const uint32_t ticket = atomicAdd(&ctl->bounds_ticket, 1u);
        s_last = ticket == gridDim.x - 1;
    }
    __syncthreads();
    if (!s_last) return;
    // the last block folds the per-block partials, all threads in parallel
    __threadfence();
    MinMax f;
    f.init();
    int all = 1;
    for (int b = threadIdx.x; b < (int)gridDim.x; b += kThreads) {
        const float *p = partials + 8 * (int64_t)b;
        for (int a = 0; a < 3; ++a) {
            f.lo[a] = min_ordered(f.lo[a], __ldcg(p + a));
            f.hi[a] = max_ordered(f.hi[a], __ldcg(p + 3 + a));
        }
        all &= __ldcg(p + 6) != 0.0f;
    }
    for (int off = 16; off > 0; off >>= 1) {
        for (int a = 0; a < 3; ++a) {
            f.lo[a] = min_ordered(f.lo[a], __shfl_xor_sync(0xffffffffu, f.lo[a], off));
            f.hi[a] = max_ordered(f.hi[a], __shfl_xor_sync(0xffffffffu, f.hi[a], off));
        }
        all &= __shfl_xor_sync(0xffffffffu, all, off);
    }
    __syncthreads();  // s_v / s_ok are reused
    if (lane == 0) {
        for (int a = 0; a < 3; ++a) {
            s_v[warp][a] = f.lo[a];
            s_v[warp][3 + a] = f.hi[a];
        }
        s_ok[warp] = all;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        float v[6];
        int ok_all = 1;
        for (int k = 0; k < 6; ++k) v[k] = s_v[0][k];
        for (int w = 1; w < kThreads / 32; ++w) {
            for (int a = 0; a < 3; ++a) {
                v[a] = min_ordered(v[a], s_v[w][a]);
                v[3 + a] = max_ordered(v[3 + a], s_v[w][3 + a]);
            }
            ok_all &= s_ok[w];
        }
        ok_all &= s_ok[0];
        for (int k = 0; k < 6; ++k) bounds[k] = v[k];
        if (!ok_all) atomicOr(&ctl->build_flags, kFlagNonfinite);
        ctl->bounds_ticket = 0;  // ready for the next reduction
    }
}

// kLayout (CodeLayout): kCodePlain writes the code alone; kCodeLow the word
// code << 32 | index (codes of at most 32 bits, for a sort that carries the
// index in the key's low half); kCodeTop the word (code >> (ib - 1)) << ib |
// index (the code's top 64 - ib bits above the index, n <= 2^ib). The
// histograms count the bytes of the code (plain, low) or of the word from
// byte top_first_byte(ib, skip) on (top): the bytes the sort's passes take
// in turn.
// kCodeHilbert: as kCodeLow with the Hilbert index of the cell, without its
// low ib bits, in place of the Morton code (the order of queries that are
// walked in packets).
__device__ const HilbertTable kHilbert = hilbert_table();

__device__ __forceinline__ void load_hilbert(uint16_t *s) {
    for (int k = threadIdx.x; k < kHilbertEntries; k += blockDim.x) s[k] = kHilbert.next[k];
}

template <int kKind, int kLayout>
__global__ void __launch_bounds__(kThreads)
    encode_kernel(const float *__restrict__ prims, int64_t n, int b, const float *__restrict__ bounds,
                  uint64_t *__restrict__ codes, uint32_t *__restrict__ hist, int passes, int ib, int skip) {
    __shared__ uint32_t s_hist[kMaxPasses * kRadix];
    for (int k = threadIdx.x; k < passes * kRadix; k += kThreads) s_hist[k] = 0;
    const Grid3 g = make_grid(bounds, b);
    const int hist_shift = kLayout == kCodeTop ? kRadixBits * top_first_byte(ib, skip) : 0;
    __shared__ uint16_t s_hilbert[kLayout == kCodeHilbert ? kHilbertEntries : 1];
    if (kLayout == kCodeHilbert) load_hilbert(s_hilbert);
    __syncthreads();
    for_each_centroid<kKind>(prims, n, [&](int64_t i, float x, float y, float z) {
        const uint64_t c = kLayout == kCodeHilbert ? hilbert(x, y, z, g, b, s_hilbert) >> ib : morton(x, y, z, g);
        const uint64_t w = kLayout == kCodeTop   ? ((c >> (ib - 1)) << ib) | (uint64_t)(uint32_t)i
                           : kLayout != kCodePlain ? (c << 32) | (uint64_t)(uint32_t)i
                                                   : c;
        codes[i] = w;
        const uint64_t h = kLayout == kCodeTop ? w >> hist_shift : c;
        for (int p = 0; p < passes; ++p)
            atomicAdd(&s_hist[p * kRadix + (uint32_t)((h >> (kRadixBits * p)) & (kRadix - 1))], 1u);
    });
    __syncthreads();
    for (int k = threadIdx.x; k < passes * kRadix; k += kThreads) {
        const uint32_t v = s_hist[k];
        if (v) atomicAdd(&hist[k], v);
    }
}

// The walk order of ray segments: word (code << 32 | i) per ray, its code the
// first 8 bits of the Hilbert index of the cell that holds the segment's
// middle (a segment longer than the scene is cut to the scene's extent, cells
// outside the scene to its border), and the histogram of the codes. *apart
// counts the runs of 32 rays whose middles are not all within an eighth of the
// scene from the first one's: where they are few, the order as given is kept.
__global__ void __launch_bounds__(kThreads)
    encode_rays_kernel(const float4 *__restrict__ rays, int64_t n, const float *__restrict__ bounds,
                       uint64_t *__restrict__ words, uint32_t *__restrict__ hist, uint32_t *apart) {
    __shared__ uint32_t s_hist[kRadix], s_apart;
    __shared__ uint16_t s_hilbert[kHilbertEntries];
    s_hist[threadIdx.x] = 0;  // kThreads == kRadix
    if (threadIdx.x == 0) s_apart = 0;
    load_hilbert(s_hilbert);
    const Grid3 g = make_grid(bounds, 3);
    const float extent = fmaxf(g.extent[0], fmaxf(g.extent[1], g.extent[2]));
    const int lane = threadIdx.x & 31;
    __syncthreads();
    for (int64_t first = (int64_t)blockIdx.x * kThreads + (threadIdx.x & ~31); first < n;
         first += (int64_t)gridDim.x * kThreads) {
        const int64_t i = min(first + lane, n - 1);
        const float4 o = rays[2 * i], d = rays[2 * i + 1];
        const float speed = fmaxf(fabsf(d.x), fmaxf(fabsf(d.y), fabsf(d.z)));
        const float t = o.w + 0.5f * fminf(d.w - o.w, extent / speed);
        const float x = o.x + t * d.x, y = o.y + t * d.y, z = o.z + t * d.z;
        const float away = fmaxf(fabsf(x - __shfl_sync(0xffffffffu, x, 0)),
                                 fmaxf(fabsf(y - __shfl_sync(0xffffffffu, y, 0)), fabsf(z - __shfl_sync(0xffffffffu, z, 0))));
        const bool together = __all_sync(0xffffffffu, away <= 0.125f * extent);
        if (lane == 0 && !together) atomicAdd(&s_apart, 1u);
        if (first + lane < n) {
            const uint64_t c = hilbert(x, y, z, g, 3, s_hilbert) >> 1;
            words[i] = c << 32 | (uint64_t)(uint32_t)i;
            atomicAdd(&s_hist[(uint32_t)c], 1u);
        }
    }
    __syncthreads();
    if (threadIdx.x == 0 && s_apart) atomicAdd(apart, s_apart);
    const uint32_t v = s_hist[threadIdx.x];
    if (v) atomicAdd(&hist[threadIdx.x], v);
}

template <int kKind>
__device__ __forceinline__ void centroid_at(const float *prims, int64_t i, float &x, float &y, float &z) {
    if (kKind == LBVH_PRIM_POINTS) {
        x = prims[3 * i];
        y = prims[3 * i + 1];
        z = prims[3 * i + 2];
    } else {
        box_centroid(prims + 6 * i, x, y, z);
    }
}

// The order of packets inside crowded cells. The Hilbert order of the queries
// has 2^levels cells per axis; where many queries share a cell (clusters far
// smaller than the scene) it says nothing about them, and a packet is 32
// queries from all over the cell: too far apart unless each of them spans most
// of it. A CTA takes a window of kWindow places; if kCrowdedPairs pairs of queries
// kCrowd places apart share a cell and are small beside it, it sorts the window by
// the curve of 17 levels (which visits the coarser cells in the same order) in
// a bitonic network, kEach places to a thread: steps inside a thread and, by
// shuffles, inside a warp, ten through shared memory. Other windows cost a look at
// one place in kCrowd.
// 2 * 10^6 queries on as many points in 64 clusters (whole call, us; before /
// now / Algorithm 1): sigma 1e-3 of the scene, 35 queries to a cell, 896 / 685 /
// 945; 1e-4, 1766 / 1026 / 1119; 1e-5, a cluster to a cell, 1761 / 1300 / 1134
// (windows are sorted one by one, so the order is as fine as 4096 queries of a
// cell allow); 16 nearest neighbours at 1e-4 9165 / 3701 / 5770.
// It is bound by instructions: 30 us for one wave of CTAs, 100 us for 2 * 10^6
// crowded queries, 3 us where nothing is crowded (20 for 2^23 queries that have to
// be looked at, 3 where one radius says that none is small). Windows of 2048: 70
// us, but the 1e-4 clusters take 1206.
constexpr int kWindow = 4096, kWindowThreads = 512, kEach = kWindow / kWindowThreads;
constexpr int kCrowd = 64, kCrowdedPairs = 4;
template <int kKind>
__global__ void __launch_bounds__(kWindowThreads)
    refine_order_kernel(QueryArgs qa, int levels, const float *__restrict__ bounds, uint32_t *order, const Control *ctl) {
    __shared__ uint64_t s_key[kWindow];
    __shared__ uint16_t s_hilbert[kHilbertEntries];
    __shared__ int s_pairs;
    if (ctl->build_flags != 0) return;  // the sort may have given up: the words are not an order
    const int t = threadIdx.x;
    const Grid3 coarse = make_grid(bounds, levels);
    const float edge = fmaxf(coarse.extent[0], fmaxf(coarse.extent[1], coarse.extent[2])) / coarse.cells;
    if (kKind == LBVH_PRIM_POINTS && !qa.radii && 4.0f * qa.radius >= edge) return;
    for (int64_t base = (int64_t)blockIdx.x * kWindow; base < qa.nq; base += (int64_t)gridDim.x * kWindow) {
        const int count = (int)min((int64_t)kWindow, qa.nq - base);
        const auto cell = [&](int at, const Grid3 &g) {
            float x, y, z;
            centroid_at<kKind>(qa.queries, (int64_t)order[base + at], x, y, z);
            return morton(x, y, z, g);
        };
        __syncthreads();  // the window before is done
        if (t == 0) s_pairs = 0;
        const bool sample = t < kWindow / kCrowd && kCrowd * t < count;
        bool small = false;
        if (sample) {
            s_key[t] = cell(kCrowd * t, coarse);
            const int64_t q = order[base + kCrowd * t];
            if (kKind == LBVH_PRIM_POINTS) {
                small = 4.0f * (qa.radii ? qa.radii[q] : qa.radius) < edge;
            } else {
                const float *b = qa.queries + 6 * q;
                small = 2.0f * fmaxf(b[3] - b[0], fmaxf(b[4] - b[1], b[5] - b[2])) < edge;
            }
        }
        __syncthreads();
        if (small && t > 0 && s_key[t] == s_key[t - 1]) atomicAdd(&s_pairs, 1);
        __syncthreads();
        if (s_pairs < kCrowdedPairs) continue;
        load_hilbert(s_hilbert);
        const Grid3 g = make_grid(bounds, 21);
        uint64_t key[kEach];  // places kEach t .. kEach t + kEach - 1: the cells of 21 levels, then their places on the curve
        uint32_t state[kEach];
#pragma unroll
        for (int j = 0; j < kEach; ++j) key[j] = cell(min(kEach * t + j, count - 1), g);
        __syncthreads();
#pragma unroll
        for (int j = 0; j < kEach; ++j) {  // as hilbert(), the steps of the places side by side: the first three bits,
            const uint32_t e = s_hilbert[2u << 6 | (uint32_t)(key[j] >> 60)];
            key[j] = key[j] << 4 | (e & 63u);
            state[j] = e & ~63u;
        }
#pragma unroll 1
        for (int k = 0; k < 10; ++k)  // then six at a time taken from the top, their places on the curve put in below
#pragma unroll
            for (int j = 0; j < kEach; ++j) {
                const uint32_t e = s_hilbert[state[j] | (uint32_t)(key[j] >> 58)];
                key[j] = key[j] << 6 | (e & 63u);
                state[j] = e & ~63u;
            }
#pragma unroll
        for (int j = 0; j < kEach; ++j) {
            const int e = kEach * t + j;
            key[j] = e < count ? key[j] >> 11 << 12 | (uint64_t)e : ~0ull;
        }
#pragma unroll 1
        for (int run = 2; run <= kWindow; run *= 2) {
            // the smaller key goes to the lower place of an ascending pair and the upper one of a descending pair
            const auto keep = [&](int j, int d, uint64_t other) {
                const int e = kEach * t + j;
                const bool smaller = ((e & d) == 0) == ((e & run) == 0);
                key[j] = (key[j] < other) == smaller ? key[j] : other;
            };
            int d = run / 2;
#pragma unroll 1
            for (; d >= kEach * 32; d /= 2) {
#pragma unroll
                for (int j = 0; j < kEach; ++j) s_key[j * kWindowThreads + t] = key[j];
                __syncthreads();
#pragma unroll
                for (int j = 0; j < kEach; ++j) keep(j, d, s_key[j * kWindowThreads + (t ^ (d / kEach))]);
                __syncthreads();
            }
#pragma unroll 1
            for (; d >= kEach; d /= 2)
#pragma unroll
                for (int j = 0; j < kEach; ++j) keep(j, d, __shfl_xor_sync(0xffffffffu, key[j], d / kEach));
#pragma unroll
            for (int c = kEach / 2; c > 0; c /= 2)
                if (c < run) {
#pragma unroll
                    for (int j = 0; j < kEach; ++j)
                        if ((j & c) == 0) {
                            const uint64_t lo = key[j], hi = key[j | c];
                            keep(j, c, hi);
                            keep(j | c, c, lo);
                        }
                }
        }
        uint32_t mine[kEach];
#pragma unroll
        for (int j = 0; j < kEach; ++j)
            mine[j] = kEach * t + j < count ? order[base + (int)(key[j] & (kWindow - 1))] : 0u;
        __syncthreads();  // every place has been read
#pragma unroll
        for (int j = 0; j < kEach; ++j)
            if (kEach * t + j < count) order[base + kEach * t + j] = mine[j];
    }
}

// The codes of the primitives in sorted order: codes[i] = the code of
// primitive perm[i] (a gather through the permutation and the same encoding).
template <int kKind>
__global__ void __launch_bounds__(kThreads)
    sorted_codes_kernel(const float *__restrict__ prims, const uint32_t *__restrict__ perm, int64_t n, int b,
                        const float *__restrict__ bounds, uint64_t *__restrict__ codes) {
    const Grid3 g = make_grid(bounds, b);
    for (int64_t i = (int64_t)blockIdx.x * kThreads + threadIdx.x; i < n; i += (int64_t)gridDim.x * kThreads) {
        const int64_t p = perm[i];
        float x, y, z;
        if (kKind == LBVH_PRIM_POINTS) {
            x = prims[3 * p];
            y = prims[3 * p + 1];
            z = prims[3 * p + 2];
        } else {
            box_centroid(prims + 6 * p, x, y, z);
        }
        codes[i] = morton(x, y, z, g);
    }
}

// ---- batches: one CTA per chunk of one instance

template <int kKind>
__global__ void __launch_bounds__(kThreads)
    batch_bounds_kernel(const float *__restrict__ prims, const BatchChunk *__restrict__ chunks,
                        float *__restrict__ partials) {
    const BatchChunk c = chunks[blockIdx.x];
    MinMax m;
    m.init();
    for (int64_t i = c.begin + threadIdx.x; i < c.end; i += kThreads) {
        float x, y, z;
        centroid_at<kKind>(prims, i, x, y, z);
        m.add(x, y, z);
    }
    __shared__ float s_v[kThreads / 32][6];
    __shared__ int s_ok[kThreads / 32];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    int ok = m.ok;
    for (int off = 16; off > 0; off >>= 1) {
        for (int a = 0; a < 3; ++a) {
            m.lo[a] = min_ordered(m.lo[a], __shfl_xor_sync(0xffffffffu, m.lo[a], off));
            m.hi[a] = max_ordered(m.hi[a], __shfl_xor_sync(0xffffffffu, m.hi[a], off));
        }
        ok &= __shfl_xor_sync(0xffffffffu, ok, off);
    }
    if (lane == 0) {
        for (int a = 0; a < 3; ++a) {
            s_v[warp][a] = m.lo[a];
            s_v[warp][3 + a] = m.hi[a];
        }
        s_ok[warp] = ok;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        float v[6];
        int all = 1;
        for (int k = 0; k < 6; ++k) v[k] = s_v[0][k];
        for (int w = 0; w < kThreads / 32; ++w) {
            for (int a = 0; a < 3; ++a) {
                v[a] = min_ordered(v[a], s_v[w][a]);
                v[3 + a] = max_ordered(v[3 + a], s_v[w][3 + a]);
            }
            all &= s_ok[w];
        }
        float *out = partials + 8 * (int64_t)blockIdx.x;
        for (int k = 0; k < 6; ++k) out[k] = v[k];
        out[6] = all ? 1.0f : 0.0f;
    }
}

__global__ void __launch_bounds__(kThreads)
    batch_bounds_fold_kernel(const float *__restrict__ partials, const int64_t *__restrict__ chunk_first,
                             int count, float *__restrict__ bounds, Control *ctl) {
    const int b = blockIdx.x * kThreads + threadIdx.x;
    if (b >= count) return;
    float v[6] = {FLT_MAX, FLT_MAX, FLT_MAX, -FLT_MAX, -FLT_MAX, -FLT_MAX};
    int all = 1;
    for (int64_t c = chunk_first[b]; c < chunk_first[b + 1]; ++c) {
        const float *p = partials + 8 * c;
        for (int a = 0; a < 3; ++a) {
            v[a] = min_ordered(v[a], p[a]);
            v[3 + a] = max_ordered(v[3 + a], p[3 + a]);
        }
        all &= p[6] != 0.0f;
    }
    for (int k = 0; k < 6; ++k) bounds[6 * (int64_t)b + k] = v[k];
    if (!all) atomicOr(&ctl->build_flags, kFlagNonfinite);
}

template <int kKind, bool kCurve>
__global__ void __launch_bounds__(kThreads)
    batch_encode_kernel(const float *__restrict__ data, const BatchChunk *__restrict__ chunks, int b,
                        const float *__restrict__ bounds, uint64_t *__restrict__ keys,
                        uint32_t *__restrict__ hist) {
    __shared__ uint32_t s_hist[kRadix];
    s_hist[threadIdx.x] = 0;  // kThreads == kRadix
    const BatchChunk c = chunks[blockIdx.x];
    const Grid3 g = make_grid(bounds + 6 * (int64_t)c.inst, b);
    __shared__ uint16_t s_hilbert[kCurve ? kHilbertEntries : 1];
    if (kCurve) load_hilbert(s_hilbert);
    __syncthreads();
    for (int64_t i = c.begin + threadIdx.x; i < c.end; i += kThreads) {
        float x, y, z;
        centroid_at<kKind>(data, i, x, y, z);
        const uint64_t key = kCurve ? hilbert(x, y, z, g, b, s_hilbert) >> 1 : morton(x, y, z, g);
        keys[i] = key;
        atomicAdd(&s_hist[(uint32_t)key & (kRadix - 1)], 1u);
    }
    __syncthreads();
    const uint32_t v = s_hist[threadIdx.x];
    if (v) atomicAdd(&hist[(int64_t)c.inst * kRadix + threadIdx.x], v);
}

}  // namespace

void launch_batch_bounds(const float *prims, int kind, const BatchTables &bt, float *partials,
                         float *bounds, Control *ctl, cudaStream_t s) {
    if (bt.nchunks <= 0) return;
    if (kind == LBVH_PRIM_POINTS)
        batch_bounds_kernel<LBVH_PRIM_POINTS><<<(unsigned)bt.nchunks, kThreads, 0, s>>>(prims, bt.chunks, partials);
    else
        batch_bounds_kernel<LBVH_PRIM_BOXES><<<(unsigned)bt.nchunks, kThreads, 0, s>>>(prims, bt.chunks, partials);
    batch_bounds_fold_kernel<<<(unsigned)((bt.count + kThreads - 1) / kThreads), kThreads, 0, s>>>(
        partials, bt.chunk_first, bt.count, bounds, ctl);
    count_launches(2);
}

void launch_batch_encode(const float *data, int kind, bool queries, const BatchTables &bt, int bits,
                         const float *bounds, uint64_t *keys, uint32_t *hist, cudaStream_t s, bool hilbert) {
    const int64_t nchunks = queries ? bt.nqchunks : bt.nchunks;
    const BatchChunk *chunks = queries ? bt.qchunks : bt.chunks;
    if (nchunks <= 0) return;
    const int b = hilbert ? 11 : bits / 3;
    const bool points = kind == LBVH_PRIM_POINTS;
    auto k = hilbert ? (points ? batch_encode_kernel<LBVH_PRIM_POINTS, true> : batch_encode_kernel<LBVH_PRIM_BOXES, true>)
                     : (points ? batch_encode_kernel<LBVH_PRIM_POINTS, false>
                               : batch_encode_kernel<LBVH_PRIM_BOXES, false>);
    k<<<(unsigned)nchunks, kThreads, 0, s>>>(data, chunks, b, bounds, keys, hist);
    count_launches(1);
}

int bounds_blocks(int64_t n) {
    const int64_t want = (n / 4 + kThreads - 1) / kThreads;
    const int64_t cap = (int64_t)device_sm_count() * 8;
    return (int)(want < 1 ? 1 : (want > cap ? cap : want));
}

void launch_bounds(const float *prims, int64_t n, int kind, float *partials, float *bounds,
                   Control *ctl, cudaStream_t s) {
    const int blocks = bounds_blocks(n);
    if (kind == LBVH_PRIM_POINTS)
        bounds_kernel<LBVH_PRIM_POINTS><<<blocks, kThreads, 0, s>>>(prims, n, partials, bounds, ctl);
    else
        bounds_kernel<LBVH_PRIM_BOXES><<<blocks, kThreads, 0, s>>>(prims, n, partials, bounds, ctl);
    count_launches(1);
}

void launch_encode(const float *prims, int64_t n, int kind, int bits, const float *bounds,
                   uint64_t *codes, uint32_t *hist, int hist_passes, int layout, int index_bits, cudaStream_t s,
                   int skip) {
    const int blocks = bounds_blocks(n);
    const int b = bits / 3;
    using Kernel = void (*)(const float *, int64_t, int, const float *, uint64_t *, uint32_t *, int, int, int);
    static const Kernel table[2][4] = {
        {encode_kernel<LBVH_PRIM_POINTS, kCodePlain>, encode_kernel<LBVH_PRIM_POINTS, kCodeLow>,
         encode_kernel<LBVH_PRIM_POINTS, kCodeTop>, encode_kernel<LBVH_PRIM_POINTS, kCodeHilbert>},
        {encode_kernel<LBVH_PRIM_BOXES, kCodePlain>, encode_kernel<LBVH_PRIM_BOXES, kCodeLow>,
         encode_kernel<LBVH_PRIM_BOXES, kCodeTop>, encode_kernel<LBVH_PRIM_BOXES, kCodeHilbert>}};
    table[kind == LBVH_PRIM_POINTS ? 0 : 1][layout]<<<blocks, kThreads, 0, s>>>(prims, n, b, bounds, codes, hist,
                                                                               hist_passes, index_bits, skip);
    count_launches(1);
}

void launch_encode_rays(const float *rays, int64_t n, const float *bounds, uint64_t *words, uint32_t *hist,
                        uint32_t *apart, cudaStream_t s) {
    encode_rays_kernel<<<bounds_blocks(n), kThreads, 0, s>>>(reinterpret_cast<const float4 *>(rays), n, bounds, words,
                                                            hist, apart);
    count_launches(1);
}

void launch_refine_order(const QueryArgs &q, int levels, const float *bounds, uint32_t *order, const Control *ctl,
                         cudaStream_t s) {
    if (q.nq <= 0) return;
    auto k = q.qkind == LBVH_Q_SPHERE ? refine_order_kernel<LBVH_PRIM_POINTS> : refine_order_kernel<LBVH_PRIM_BOXES>;
    const int64_t windows = (q.nq + kWindow - 1) / kWindow, most = 4 * (int64_t)device_sm_count();
    k<<<(unsigned)(windows < most ? windows : most), kWindowThreads, 0, s>>>(q, levels, bounds, order, ctl);
    count_launches(1);
}

void launch_sorted_codes(const float *prims, const uint32_t *perm, int64_t n, int kind, int bits,
                         const float *bounds, uint64_t *codes, cudaStream_t s) {
    if (n <= 0) return;
    int64_t blocks = (n + kThreads - 1) / kThreads;
    const int64_t cap = (int64_t)device_sm_count() * 16;
    if (blocks > cap) blocks = cap;
    if (kind == LBVH_PRIM_POINTS)
        sorted_codes_kernel<LBVH_PRIM_POINTS><<<(unsigned)blocks, kThreads, 0, s>>>(prims, perm, n, bits / 3,
                                                                                    bounds, codes);
    else
        sorted_codes_kernel<LBVH_PRIM_BOXES><<<(unsigned)blocks, kThreads, 0, s>>>(prims, perm, n, bits / 3,
                                                                                   bounds, codes);
    count_launches(1);
}

}  // namespace lbvh
