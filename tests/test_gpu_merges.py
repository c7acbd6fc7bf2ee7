"""The bottom-up pass by merges (nodes of a group of leaves formed side by
side, then what the groups left, in further merges or by climbing) against the
Karras build of the same primitives: every field of the tree, at the edges of
the groups and of the rules that say how far the merges go, and for chains of
leaves that leave more over than a group's slots hold."""
from __future__ import annotations

import numpy as np
import pytest

from paper_2402_00665_gb300 import _build, inputs

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


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


def karras(prims, kind, bits):
    t = L().Tree().build(prims, kind, bits, algorithm=L().BUILD_KARRAS)
    e = t.export()
    t.close()
    return e


def same(got, want):
    for k in want:
        a, b = np.asarray(got[k]), np.asarray(want[k])
        assert a.tobytes() == b.tobytes(), k


def chain(before, after, seed):
    """`before` points, 60 points whose codes have one bit each below the
    common octant (their gaps grow along the sorted order), `after` points."""
    rng = np.random.default_rng(seed)
    cell = 2.0 ** -21
    low = rng.random((before, 3)) * [0.5, 1.0, 1.0]
    low[0] = 0.0
    links = np.full((61, 3), 0.5)
    for k in range(60):
        links[k + 1, 2 - k % 3] += cell * (1 << (k // 3))
    top = 0.5 + 0.5 * rng.random((after, 3))
    top[-1] = 1.0
    return np.concatenate([low, links, top]).astype(np.float32)


@pytest.mark.parametrize("kind", ["points", "boxes"])
@pytest.mark.parametrize("n", [1, 2, 31, 32, 33, 127, 128, 129, 1023, 1025, 5119, 5121, 24576, 24577, 131073, 4194304, 4194305])
def test_group_edges(n, kind):
    lbvh = L()
    pts = inputs.uniform_points(n, seed=n)
    prims = pts if kind == "points" else np.concatenate([pts, pts + np.float32(0.01)], axis=1)
    code = lbvh.POINTS if kind == "points" else lbvh.BOXES
    prims = torch.from_numpy(prims).cuda()
    t = lbvh.Tree().build(prims, code, 63)
    e = t.export()
    same(e, karras(prims, code, 63))
    s = lbvh.Tree().build_from_sorted(e["sorted"], e["perm"], prims, code)
    got = s.export()
    same({k: v for k, v in got.items() if k != "bounds"}, {k: v for k, v in e.items() if k != "bounds"})
    s.close()
    t.close()


@pytest.mark.parametrize("before", [1152 - 5, 1152 - 20, 1152 - 45, 70000])
def test_lists_longer_than_their_slots(before):
    lbvh = L()
    for copies in (1, 200):  # 200: every gap of the chain between runs of equal codes
        pts = np.repeat(chain(before, 300, seed=before), copies if before < 5000 else 1, axis=0)
        t = lbvh.Tree().build(pts, lbvh.POINTS, 63)
        same(t.export(), karras(pts, lbvh.POINTS, 63))
        t.close()


def test_batch_of_chains_and_small_instances():
    lbvh = L()
    parts = [chain(b, a, seed=b) for b, a in ((1152 - 5, 300), (40, 3), (1000, 1), (3000, 7000))]
    parts += [inputs.uniform_points(n, seed=n) for n in (1, 1, 2, 3, 130, 1, 2, 20000, 1)]
    off = np.concatenate([[0], np.cumsum([len(p) for p in parts])]).astype(np.int64)
    batch = lbvh.Batch()
    batch.build_query(torch.from_numpy(np.concatenate(parts)).cuda(), off, lbvh.POINTS, 63)
    for k, p in enumerate(parts):
        same(batch.export(k), karras(p, lbvh.POINTS, 63))
    batch.close()
