"""Packets that are cut up. Into two halves, the second of which gives up: the
first half keeps what it has taken, and only the second half's lanes are left
over (one warp runs the walk itself over hand-made leaf blocks). Into shapes:
box queries that are long along different axes have the hits of Algorithm 1,
and take no more than about its time."""
from __future__ import annotations

import subprocess

import numpy as np
import pytest

from paper_2402_00665_gb300 import _build, inputs

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


NODES = 4  # walk variant: Algorithm 1, one thread per query


def rods(n, length, thick, seed):
    """float32[n, 6]: boxes long along one random axis, every 97th an infinite slab, every 101st a NaN."""
    rng = np.random.default_rng(seed)
    half = np.full((n, 3), thick / 2)
    half[np.arange(n), rng.integers(0, 3, n)] = length / 2
    c = rng.random((n, 3))
    box = np.concatenate([c - half, c + half], axis=1).astype(np.float32)
    box[::97, 0], box[::97, 3] = -np.inf, np.inf
    box[::101, 2] = np.nan
    return box


def walk_ms(tree, q, offsets, hits):
    from paper_2402_00665_gb300 import lbvh
    best = 1e9
    for _ in range(6):
        st, _ = tree.query_into(q, lbvh.BOX, offsets, hits)
        assert st == lbvh.OK
        best = min(best, tree.stage_times()["query_walk"])
    return best


@pytest.mark.parametrize("kind", ["points", "boxes", "rods"])
def test_shapes(kind):
    from paper_2402_00665_gb300 import lbvh
    n, nq = 300_000, 200_003  # more than 800 queries per SM: packets
    pts = inputs.uniform_points(n, seed=7)
    prims = {"points": pts, "boxes": np.concatenate([pts, pts + np.float32(1e-4)], axis=1),
             "rods": np.nan_to_num(rods(n, 0.02, 0.002, seed=8), nan=0.5, posinf=1.0, neginf=0.0)}[kind]
    tree = lbvh.Tree().build(prims, lbvh.POINTS if kind == "points" else lbvh.BOXES, 63)
    q = torch.from_numpy(rods(nq, 0.2, 0.002, seed=9)).cuda()
    got = [x.cpu() for x in tree.query(q, lbvh.BOX)]
    tree.set_tuning(-1, NODES)
    want = [x.cpu() for x in tree.query(q, lbvh.BOX)]
    assert torch.equal(got[0], want[0]) and torch.equal(got[1], want[1])
    off = np.array([0, 1000, n // 2, n], np.int64)
    qoff = np.array([0, 5, nq // 2, nq], np.int64)
    if kind == "points":  # the same in a batch of three trees
        batch = lbvh.Batch()
        o, h, total, st = batch.build_query(tree._keep, off, lbvh.POINTS, 63, queries=q, query_offsets=qoff,
                                            qkind=lbvh.BOX, capacity=4 * got[1].numel())
        assert st == lbvh.OK
        o, h = o.cpu(), h[:total].cpu()
        for k in range(3):
            one = lbvh.Tree().build(pts[off[k]:off[k + 1]], lbvh.POINTS, 63)
            one.set_tuning(-1, NODES)
            wo, wh = [x.cpu() for x in one.query(q[qoff[k]:qoff[k + 1]], lbvh.BOX)]
            assert torch.equal(o[qoff[k]:qoff[k + 1] + 1] - o[qoff[k]], wo)
            assert torch.equal(h[o[qoff[k]]:o[qoff[k + 1]]], wh)
            one.close()
        batch.close()
    tree.close()


def test_shapes_take_no_longer_than_the_nodes():
    """Packets that read the region of unlike rods as a whole took 5 times as long."""
    from paper_2402_00665_gb300 import lbvh
    n = 300_000
    tree = lbvh.Tree().build(inputs.uniform_points(n, seed=7), lbvh.POINTS, 63)
    q = rods(n, 0.2, 0.002, seed=9)
    q[::97] = q[1]
    q[::101] = q[1]
    q = torch.from_numpy(q).cuda()
    off, hits = tree.query(q, lbvh.BOX)
    tree.set_profiling(True)
    packets = walk_ms(tree, q, off, hits)
    tree.set_tuning(-1, NODES)
    nodes = walk_ms(tree, q, off, hits)
    tree.close()
    assert packets < 3 * nodes, (packets, nodes)
