"""Nearest neighbours among many primitives at the same distance (copies of a
point, boxes around the query): rows as by the heap over the nodes, which larger k
take, and, where packets end up with more ties than they keep, in no more than
twice its time."""
from __future__ import annotations

import numpy as np
import pytest

from paper_2402_00665_gb300 import _build

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module", autouse=True)
def lib():
    if not torch.cuda.is_available():
        pytest.skip("needs a GPU")
    _build.build()
    from paper_2402_00665_gb300 import lbvh
    return lbvh.load()


@pytest.mark.parametrize("kind", ["points", "boxes"])
@pytest.mark.parametrize("k", [3, 5, 8, 16, 17, 32])
@pytest.mark.parametrize("copies", [1, 7, 8, 33, 64, 65, 100, 1000])
@pytest.mark.parametrize("own", [True, False])
def test_copies(kind, k, copies, own):
    from paper_2402_00665_gb300 import lbvh
    n = 20_011
    rng = np.random.default_rng(copies)
    at = rng.random((n // copies + 1, 3)).astype(np.float32)
    pts = np.repeat(at, copies, axis=0)[:n]
    pts = pts[rng.permutation(n)]  # indices of copies lie apart
    q = pts if own else at[rng.integers(0, len(at), n)]
    prims = pts if kind == "points" else np.concatenate([pts - 0.05, pts + 0.05], axis=1)
    prims, q = torch.from_numpy(prims).cuda(), torch.from_numpy(np.ascontiguousarray(q)).cuda()
    tree = lbvh.Tree().build(prims, lbvh.POINTS if kind == "points" else lbvh.BOXES, 63)
    q = prims if own and kind == "points" else q
    idx, d2 = tree.knn(q, k)
    widx, wd2 = tree.knn(q, 40)  # the heap
    assert torch.equal(idx, widx[:, :k]) and torch.equal(d2, wd2[:, :k])
    tree.close()


def test_a_lattice_takes_no_longer_than_the_heap():
    """With bounds that are distances alone it took 4 times as long."""
    from paper_2402_00665_gb300 import lbvh
    lib = lbvh.load()
    p = (torch.rand((2_000_000, 3), generator=torch.Generator(device="cuda").manual_seed(1), device="cuda") * 30).floor()
    tree = lbvh.Tree().build(p, lbvh.POINTS, 63)
    want = tree.knn(p, 16)
    tree.set_profiling(True)

    def ms():
        best = 1e9
        for _ in range(5):
            got = tree.knn(p, 16)
            best = min(best, tree.stage_times()["query_walk"])
            assert torch.equal(got[0], want[0]) and torch.equal(got[1], want[1])
        return best

    packets = ms()
    tree.close()
    tree = lbvh.Tree().build(p, lbvh.POINTS, 63)
    tree.set_profiling(True)
    tree.check()
    assert lib.lbvh_test_limit_allocation(1 << 20) == lbvh.OK  # no room for packets' scratch
    try:
        heap = ms()
    finally:
        assert lib.lbvh_test_limit_allocation(0) == lbvh.OK
    tree.close()
    assert packets < 2 * heap, (packets, heap)
