"""A packet that was cut in two, whose second half then gives up: the first
half keeps what it has taken, and only the second half's lanes are left over.
One warp runs the walk itself over hand-made leaf blocks."""
from __future__ import annotations

import subprocess

import pytest

from paper_2402_00665_gb300 import _build

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

# 64 points: the leaf block b holds 8 at x = b (b > 0: x = 9 + b). Lanes 0..15
# ask for a ball of radius 1/2 around x = 0 (block 0, 8 hits), lanes 16..31 for
# one of radius 5 around x = 13 (blocks 1..7, more than kMaxBlocks).
PROGRAM = r"""
#include <cstdio>
#include <cstring>
#include "packet.cuh"
using namespace lbvh;
struct Counter {
    static constexpr int kMaxBlocks = 4;
    uint32_t cnt;
    __device__ bool full() const { return false; }
    __device__ void reset() { cnt = 0; }
    template <int kP, typename Q>
    __device__ void take(uint32_t m, const PacketSmem<kP> &, int, const Q &) { cnt += __popc(m); }
};
__global__ void run(const float4 *leaves, const float4 *rec, uint32_t *counts, uint32_t *left) {
    __shared__ PacketSmem<LBVH_PRIM_POINTS> sm;
    const int lane = threadIdx.x;
    const Sphere q{make_float3(lane < 16 ? 0.f : 13.f, 0.f, 0.f), lane < 16 ? 0.25f : 25.f};
    Counter k{0u};
    const uint32_t l = packets<LBVH_Q_SPHERE, LBVH_PRIM_POINTS>(Blocks{leaves, rec, 64, 1u}, sm, q, kFull, k);
    counts[lane] = k.cnt;
    if (lane == 0) *left = l;
}
int main() {
    float4 leaves[64], rec[18];
    auto x = [](int b) { return b ? 9.f + b : 0.f; };
    const uint32_t exists = kBlockExists;
    float w;
    std::memcpy(&w, &exists, 4);
    for (int i = 0; i < 64; ++i) {
        const uint32_t id = i;
        leaves[i] = make_float4(x(i / 8), 0.f, 0.f, 0.f);
        std::memcpy(&leaves[i].w, &id, 4);
    }
    rec[0] = make_float4(0.f, 0.f, 0.f, 0.f);
    rec[1] = make_float4(16.f, 0.f, 0.f, w);
    for (int b = 0; b < 8; ++b) {
        rec[2 + 2 * b] = make_float4(x(b), 0.f, 0.f, 0.f);
        rec[3 + 2 * b] = make_float4(x(b), 0.f, 0.f, w);
    }
    float4 *dl, *dr;
    uint32_t *out, host[33];
    if (cudaMalloc(&dl, sizeof leaves) || cudaMalloc(&dr, sizeof rec) || cudaMalloc(&out, sizeof host)) return 2;
    cudaMemcpy(dl, leaves, sizeof leaves, cudaMemcpyHostToDevice);
    cudaMemcpy(dr, rec, sizeof rec, cudaMemcpyHostToDevice);
    run<<<1, 32>>>(dl, dr, out, out + 32);
    if (cudaMemcpy(host, out, sizeof host, cudaMemcpyDeviceToHost) != cudaSuccess) return 3;
    for (uint32_t v : host) std::printf("%u ", v);
    return 0;
}
"""


def test_first_half_keeps_its_hits(tmp_path):
    if not torch.cuda.is_available():
        pytest.skip("needs a GPU")
    src, exe = tmp_path / "split.cu", tmp_path / "split"
    src.write_text(PROGRAM)
    subprocess.run([_build.nvcc(), *_build.ARCH, *_build.FLAGS, str(src), "-o", str(exe)], check=True)
    out = subprocess.run([str(exe)], capture_output=True, text=True)
    assert out.returncode == 0, (out.returncode, out.stdout, out.stderr)
    *counts, left = [int(v) for v in out.stdout.split()]
    assert left == 0xFFFF0000
    assert counts[:16] == [8] * 16
