"""Range queries through the leaf blocks (packets of 32 queries, 8 lanes per
query) against Algorithm 1 over the nodes, which walk variant 4 runs: the same
CSR bit for bit at the edges of the blocks' levels, for every query and
primitive kind, with special queries, queries too far apart for a packet, and
after the leaves changed."""
from __future__ import annotations

import numpy as np
import pytest

from paper_2402_00665_gb300 import _build, inputs

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

NODES = 4  # walk variant: Algorithm 1, one thread per query
PACKETS = 100_003  # queries, enough for packets whatever the order


@pytest.fixture(scope="module", autouse=True)
def lib():
    if not torch.cuda.is_available():
        pytest.skip("needs a GPU")
    _build.build()
    from paper_2402_00665_gb300 import lbvh
    return lbvh.load()


def L():
    from paper_2402_00665_gb300 import lbvh
    return lbvh


def csr(tree, q, qkind, **kw):
    off, hits = tree.query(q, qkind, **kw)
    return off.cpu().numpy(), hits.cpu().numpy()


def both(tree, q, qkind, **kw):
    tree.set_tuning(-1, -1)
    got = csr(tree, q, qkind, **kw)
    tree.set_tuning(-1, NODES)
    want = csr(tree, q, qkind, **kw)
    tree.set_tuning(-1, -1)
    assert np.array_equal(got[0], want[0])
    assert np.array_equal(got[1], want[1])
    return want


def boxes_at(points, half):
    return np.concatenate([points - half, points + half], axis=1).astype(np.float32)


@pytest.mark.parametrize("nq", [37, PACKETS])
@pytest.mark.parametrize("kind", ["points", "boxes"])
@pytest.mark.parametrize("n", [1, 2, 7, 8, 9, 63, 64, 65, 511, 512, 513, 4095, 4096, 4097, 32767, 32769, 262145])
def test_block_levels(n, kind, nq):
    lbvh = L()
    pts = inputs.uniform_points(n, seed=n)
    q = inputs.uniform_points(nq, seed=n + 1)
    r = 0.6 * float(inputs.radius_for_neighbours(n))
    t = lbvh.Tree()
    t.build(pts if kind == "points" else boxes_at(pts, 0.2 * r), lbvh.POINTS if kind == "points" else lbvh.BOXES, 63)
    total = both(t, q, lbvh.SPHERE, radius=r)[0][-1]
    both(t, boxes_at(q, 0.7 * r), lbvh.BOX)
    assert total > 0 or n * nq < 1000
    t.close()


@pytest.mark.parametrize("nq", [900, PACKETS])
def test_special_queries(nq):
    lbvh = L()
    n = 5000
    pts = inputs.uniform_points(n, seed=3)
    q = inputs.uniform_points(nq, seed=4)
    radii = np.full(nq, 0.03, np.float32)
    inf, nan = np.float32(np.inf), np.float32(np.nan)
    q[5::97, 1], q[6::97, 0], q[7::97, 2] = nan, inf, -inf
    radii[8::97], radii[9::97], radii[10::97], radii[11::97] = nan, 0.0, -0.05, 3e38
    radii[12::9973] = inf
    q[11::194, 2], q[12::9973, 0] = inf, -inf  # an infinite distance within an infinite radius
    t = lbvh.Tree().build(pts, lbvh.POINTS, 30)
    both(t, q, lbvh.SPHERE, radii=radii)
    b = boxes_at(q, 0.03)
    b[13::97, :3], b[14::97, 3:] = b[13::97, 3:] + 0.01, nan  # the wrong way round, and NaN
    both(t, b, lbvh.BOX)
    t.close()


@pytest.mark.parametrize("n,scale", [(300_000, 0.02), (300_000, 1.5), (20_000, 12.0)])
def test_queries_far_apart_and_long_lists(n, scale):
    """Regions that are not tight (small radii), lists past a slot (large ones), and jumps between clusters."""
    lbvh = L()
    pts = inputs.gaussian_mixture_points(n, seed=7, components=5, sigma=0.02)
    q = np.concatenate([inputs.gaussian_mixture_points(PACKETS - 2000, seed=7, components=5, sigma=0.05),
                        inputs.uniform_points(2000, seed=8)])
    r = scale * float(inputs.radius_for_neighbours(n)) * 0.1
    t = lbvh.Tree().build(pts, lbvh.POINTS, 63)
    off, _ = both(t, q, lbvh.SPHERE, radius=r)
    if scale > 10:
        assert np.diff(off).max() > 64
    t.close()


def test_own_points_and_changed_leaves():
    lbvh = L()
    n = 120_001
    pts = torch.from_numpy(inputs.uniform_points(n, seed=11)).cuda()
    r = float(inputs.radius_for_neighbours(n))
    t = lbvh.Tree().build(pts, lbvh.POINTS, 30)
    first = both(t, pts, lbvh.SPHERE, radius=r)
    moved = pts + 0.5 * r * torch.randn_like(pts)
    t.refit(moved)
    second = both(t, moved, lbvh.SPHERE, radius=r)
    assert first[0][-1] != second[0][-1]
    image = t.save()
    loaded = lbvh.Tree().load(image)
    off, hits = csr(loaded, moved, lbvh.SPHERE, radius=r)
    assert np.array_equal(off, second[0]) and np.array_equal(hits, second[1])
    t.build(pts[:5000].contiguous(), lbvh.POINTS, 30, algorithm=lbvh.BUILD_KARRAS)
    both(t, pts, lbvh.SPHERE, radius=4 * r)
    t.close()
    loaded.close()


def test_batch_of_small_and_empty_instances():
    """Warps whose queries belong to several instances."""
    lbvh = L()
    sizes = np.array([0, 1, 5, 31, 32, 33, 0, 64, 65, 300, 1, 1, 4097, 9000, 2], np.int64)
    off = np.concatenate([[0], np.cumsum(sizes)]).astype(np.int64)
    pts = inputs.uniform_points(int(off[-1]), seed=31)
    q = inputs.uniform_points(int(off[-1]), seed=32)
    batch = lbvh.Batch()
    boff, bhits, total, st = batch.build_query(torch.from_numpy(pts).cuda(), off, lbvh.POINTS, 30,
                                               torch.from_numpy(q).cuda(), off, radius=0.08, capacity=4_000_000)
    assert st == lbvh.OK
    boff, bhits = boff.cpu().numpy(), bhits.cpu().numpy()
    for k, n in enumerate(sizes):
        a, e = off[k], off[k + 1]
        if n == 0:
            continue
        t = lbvh.Tree().build(pts[a:e], lbvh.POINTS, 30)
        t.set_tuning(-1, NODES)
        o, h = csr(t, q[a:e], lbvh.SPHERE, radius=0.08)
        assert np.array_equal(boff[a:e + 1] - boff[a], o)
        assert np.array_equal(bhits[boff[a]:boff[e]], h)
        t.close()
    batch.close()


def knn_both(tree, q, k):
    """k nearest in packets (all queries at once), by 8 lanes per query (pieces too small for packets) and one
    thread per query (the first columns of 33 neighbours, more than the others take)."""
    idx, d2 = tree.knn(q, k)
    step = 5000
    few = [tree.knn(q[a:a + step], k) for a in range(0, len(q), step)]
    assert torch.equal(idx, torch.cat([w[0] for w in few]))
    assert torch.equal(d2, torch.cat([w[1] for w in few]))
    want = tree.knn(q, 33)
    assert torch.equal(idx, want[0][:, :k])
    assert torch.equal(d2, want[1][:, :k])


@pytest.mark.parametrize("kind", ["points", "boxes"])
@pytest.mark.parametrize("k", [1, 3, 4, 5, 8, 9, 16, 17, 32])
def test_knn_packets_other_queries(k, kind):
    lbvh = L()
    nq = 40_001
    for n in (1024, 4097, 60_001):
        pts = inputs.gaussian_mixture_points(n, seed=n + k, components=6, sigma=0.05)
        q = np.concatenate([inputs.gaussian_mixture_points(nq - 3000, seed=n + k, components=6, sigma=0.06),
                            inputs.uniform_points(3000, seed=k)])
        q[7::991, 0], q[8::991, 1], q[9::991, 2] = np.nan, np.inf, -np.inf
        t = lbvh.Tree().build(pts if kind == "points" else boxes_at(pts, 0.002),
                              lbvh.POINTS if kind == "points" else lbvh.BOXES, 63 if n > 5000 else 30)
        knn_both(t, torch.from_numpy(q).cuda(), k)
        t.close()


@pytest.mark.parametrize("k", [2, 16, 31])
def test_knn_packets_own_points_ties_and_duplicates(k):
    lbvh = L()
    for pts in (inputs.uniform_points(30_011, seed=1), inputs.duplicated_points(30_011, 700, seed=2),
                np.round(inputs.uniform_points(30_011, seed=3) * 24).astype(np.float32),  # a lattice: equal distances
                np.full((12_000, 3), 0.5, np.float32)):
        p = torch.from_numpy(pts).cuda()
        t = lbvh.Tree().build(p, lbvh.POINTS, 63)
        knn_both(t, p, k)
        t.close()


def test_knn_packets_in_chunks_without_distances():
    lbvh = L()
    n = (1 << 20) + 77  # more than one chunk of queries
    p = torch.from_numpy(inputs.uniform_points(n, seed=4)).cuda()
    t = lbvh.Tree().build(p, lbvh.POINTS, 30)
    idx, none = t.knn(p, 8, distances=False)
    assert none is None
    for a in (0, 524_288, n - 3000):
        assert torch.equal(idx[a:a + 3000], t.knn(p[a:a + 3000].contiguous(), 8)[0])
    t.close()


@pytest.mark.parametrize("nq", [4095, 4096, 30_001])
def test_ray_order(nq):
    """Rays are walked by cells of their middles: pieces too small for an order give the same lists, with parallel
    axes, reversed, unbounded and non-finite segments among them."""
    lbvh = L()
    n = 20_000
    t = lbvh.Tree().build(boxes_at(inputs.uniform_points(n, seed=1), 0.01), lbvh.BOXES, 63)
    rays = inputs.random_rays(nq, seed=2, tmax=0.3)
    rays[3::17, 4], rays[4::17, 5:7], rays[5::31, 4:7] = 0.0, 0.0, 0.0
    rays[6::29, 7], rays[7::29, 3], rays[8::29, 7] = np.inf, -np.inf, -0.1
    rays[9::101, 0], rays[10::101, 5], rays[11::101, 7], rays[12::101, 4] = np.nan, np.inf, np.nan, 1e-42
    off, hits = csr(t, rays, lbvh.RAY)
    assert off[-1] > nq
    for a in range(0, nq, 4000):
        o, h = csr(t, rays[a:a + 4000], lbvh.RAY)
        assert np.array_equal(off[a:a + len(o)] - off[a], o)
        assert np.array_equal(hits[off[a]:off[a + len(o) - 1]], h)
    t.close()


@pytest.mark.parametrize("kind", ["points", "boxes"])
@pytest.mark.parametrize("n", [1, 8, 65, 513, 40000])
@pytest.mark.parametrize("nq", [1, 33, 5000, 50_000, 110_003])
def test_rays(n, kind, nq):
    """8 lanes per ray, with and without an order, and a thread per ray (110,003): rays with parallel axes,
    unbounded, empty and not finite."""
    lbvh = L()
    pts = inputs.uniform_points(n, seed=n)
    tree = lbvh.Tree()
    if kind == "points":  # some rays start at points, so they hit them
        tree.build(pts, lbvh.POINTS, 63)
    else:
        tree.build(boxes_at(pts, 0.02), lbvh.BOXES, 63)
    rng = np.random.default_rng(nq)
    rays = np.zeros((nq, 8), np.float32)
    rays[:, :3] = pts[rng.integers(0, n, nq)]
    rays[:, 4:7] = rng.normal(size=(nq, 3))
    rays[:, 7] = rng.random(nq)
    rays[::5, 4] = 0.0
    rays[::7, 7] = np.inf
    rays[::11, 7] = -1.0
    rays[3::97, 5] = np.nan
    both(tree, torch.from_numpy(rays).cuda(), lbvh.RAY)
    tree.close()


@pytest.mark.parametrize("bits", [3, 30, 33, 63])
@pytest.mark.parametrize("n", [1, 2, 31, 33, 1023, 1024, 1025, 4096, 4097, 8191, 8192, 8193, 16384, 16385])
def test_small_builds(n, bits):
    """Bounds, codes and sort of a small tree in one launch: the tree of the general sort (a chosen sort variant)."""
    lbvh = L()
    pts = inputs.uniform_points(n, seed=n)
    pts[: n // 3] = pts[0]  # equal codes
    if n > 40:
        pts[n // 2:, 2] = 0.5
        pts[7, 0] = -0.0
    for prims, kind in ((pts, lbvh.POINTS), (boxes_at(pts, 0.01), lbvh.BOXES)):
        got, want = lbvh.Tree(), lbvh.Tree()
        want.set_tuning(0, -1)
        got.build(prims, kind, bits).check()
        want.build(prims, kind, bits).check()
        a, b = got.export(), want.export()
        for key in ("perm", "sorted", "left", "skip_internal", "skip_leaf"):
            assert np.array_equal(a[key], b[key]), key
        for key in ("internal_box", "leaf_box", "bounds"):
            assert np.array_equal(a[key].view(np.uint32), b[key].view(np.uint32)), key
        got.close()
        want.close()


def test_small_build_refuses_non_finite_points_and_recovers():
    lbvh = L()
    pts = inputs.uniform_points(3000, seed=1)
    bad = pts.copy()
    bad[2999, 1] = np.inf
    t = lbvh.Tree().build(bad, lbvh.POINTS, 63)
    assert t.status() == lbvh.ERR_NONFINITE
    t.build(pts, lbvh.POINTS, 63).check()
    t.close()


@pytest.mark.parametrize("nq", [1, 4096, 4097, 300_001, 1_245_184, 1_245_185])
def test_scan_of_counts(nq):
    """One tile, several by look-back, and the three-pass scan: offsets against the counts' cumulative sum."""
    lbvh = L()
    pts = inputs.uniform_points(300, seed=1)
    t = lbvh.Tree().build(pts, lbvh.POINTS, 30)
    q = torch.rand((nq, 3), device="cuda")
    off, hits = t.query(q, lbvh.SPHERE, radius=0.1)
    p = torch.from_numpy(pts).cuda()
    counts = torch.cat([((a[:, None] - p[None]).double().square().sum(2) <= 0.01).sum(1) for a in q.split(20_000)])
    want = torch.cat([torch.zeros(1, dtype=torch.int64, device="cuda"), counts.cumsum(0)])
    assert int(off[-1]) == hits.numel()
    assert (off.diff() - counts).abs().sum() <= max(1, nq // 10_000)  # FP64 at the ball's edge
    assert abs(int(off[-1]) - int(want[-1])) <= max(1, nq // 10_000)
    t.close()
