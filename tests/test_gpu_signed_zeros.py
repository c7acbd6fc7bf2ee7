"""Box queries whose faces touch a primitive's at zero, with either sign of zero:
the closed overlap test is a comparison, for which -0 equals +0. Packets of
queries (many queries, batches), 8 lanes per query (few) and Algorithm 1 over
the nodes (walk variant 4) give the lists that NumPy's comparisons give."""
from __future__ import annotations

import numpy as np
import pytest

from paper_2402_00665_gb300 import _build

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

NODES = 4  # walk variant: Algorithm 1, one thread per query
VALUES = np.array([-0.0, 0.0, 0.25, -0.25, 1.0], np.float32)


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


def points(n, seed):
    return VALUES[np.random.default_rng(seed).integers(0, len(VALUES), (n, 3))]


def boxes(n, seed):
    """Ordered bounds, faces of either zero among them."""
    a, b = points(n, seed), points(n, seed + 1)
    lower = a <= b
    return np.concatenate([np.where(lower, a, b), np.where(lower, b, a)], axis=1)


def brute(prims, q):
    """Counts and concatenated lists by comparison."""
    plo, phi = prims[:, :3], prims[:, -3:]
    counts, lists = [], []
    for part in np.array_split(q, max(1, len(q) // 2000)):
        m = ((part[:, None, :3] <= phi[None]) & (plo[None] <= part[:, None, 3:])).all(axis=2)
        counts.append(m.sum(axis=1))
        lists.append(np.nonzero(m)[1])
    return np.concatenate(counts), np.concatenate(lists).astype(np.int32)


def csr(tree, q):
    off, hits = tree.query(q, L().BOX)
    return off.cpu().numpy(), hits.cpu().numpy()


@pytest.mark.parametrize("nq", [900, 130_003])  # 8 lanes per query, packets
@pytest.mark.parametrize("kind", ["points", "boxes"])
def test_box_queries_touching_at_zero(kind, nq):
    lbvh = L()
    n = 90
    prims = points(n, 1) if kind == "points" else boxes(n, 2)
    q = boxes(nq, 4)
    t = lbvh.Tree().build(prims, lbvh.POINTS if kind == "points" else lbvh.BOXES, 63)
    got = csr(t, q)
    t.set_tuning(-1, NODES)
    nodes = csr(t, q)
    counts, lists = brute(prims, q)
    assert np.array_equal(np.diff(nodes[0]), counts) and np.array_equal(nodes[1], lists)
    assert np.array_equal(got[0], nodes[0]) and np.array_equal(got[1], nodes[1])
    t.close()


@pytest.mark.parametrize("kind", ["points", "boxes"])
def test_batched_box_queries_touching_at_zero(kind):
    lbvh = L()
    sizes = np.array([1, 40, 7, 90], np.int64)
    off = np.concatenate([[0], np.cumsum(sizes)]).astype(np.int64)
    n = int(off[-1])
    prims = points(n, 11) if kind == "points" else boxes(n, 12)
    q = boxes(n, 14)
    batch = lbvh.Batch()
    boff, bhits, _, st = batch.build_query(torch.from_numpy(prims).cuda(), off,
                                           lbvh.POINTS if kind == "points" else lbvh.BOXES, 30,
                                           torch.from_numpy(q).cuda(), off, qkind=lbvh.BOX, capacity=n * n)
    assert st == lbvh.OK
    boff, bhits = boff.cpu().numpy(), bhits.cpu().numpy()
    for k in range(len(sizes)):
        a, e = off[k], off[k + 1]
        counts, lists = brute(prims[a:e], q[a:e])
        assert np.array_equal(np.diff(boff[a:e + 1]), counts)
        assert np.array_equal(bhits[boff[a]:boff[e]], lists)
    batch.close()


@pytest.mark.parametrize("n", [1, 8, 9, 65, 513, 4097, 32769])
@pytest.mark.parametrize("kind", ["points", "boxes"])
def test_box_packets(n, kind):
    """Enough box queries for packets (over 800 per SM) at the edges of the blocks' levels."""
    lbvh = L()
    rng = np.random.default_rng(n)
    half = np.float32(0.3 * n ** (-1 / 3))
    c, qc = rng.random((n, 3), np.float32), rng.random((130_003, 3), np.float32)
    prims = c if kind == "points" else np.concatenate([c - half, c + half], axis=1)
    q = np.concatenate([qc - half, qc + half], axis=1)
    t = lbvh.Tree().build(prims, lbvh.POINTS if kind == "points" else lbvh.BOXES, 63)
    got = csr(t, q)
    t.set_tuning(-1, NODES)
    want = csr(t, q)
    assert np.array_equal(got[0], want[0]) and np.array_equal(got[1], want[1])
    t.close()
