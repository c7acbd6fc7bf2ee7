"""A query order whose sort gave up a wait (a tile that never publishes) holds
words that were never written. Every kind of query on it reports
LBVH_ERR_TIMEOUT and indexes no query past the last (the rows past the last in
buffers that go on behind it stay as they were), and the next call is correct."""
from __future__ import annotations

import numpy as np
import pytest

from paper_2402_00665_gb300 import _build, inputs

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

NODES = 4  # walk variant: Algorithm 1, one thread per query


@pytest.fixture(scope="module", autouse=True)
def lib():
    if not torch.cuda.is_available():
        pytest.skip("needs a GPU")
    _build.build()
    from paper_2402_00665_gb300 import lbvh
    return lbvh.load()


@pytest.mark.parametrize("how", ["range", "nodes", "knn", "knn_heap"])
def test_order_that_gave_up(how):
    from paper_2402_00665_gb300 import lbvh
    lib = lbvh.load()
    n, nq = 60_000, 150_001
    tree = lbvh.Tree().build(inputs.uniform_points(n, seed=3), lbvh.POINTS, 30)
    tree.check()
    if how == "nodes":
        tree.set_tuning(-1, NODES)
    q = torch.from_numpy(inputs.uniform_points(nq, seed=4)).cuda()
    k = 8 if how == "knn" else 2
    beyond = 64  # rows behind the last query's, which nothing may write
    idx = torch.full((nq + beyond, k), 7, dtype=torch.int32, device="cuda")
    d2 = torch.full((nq + beyond, k), 7.0, device="cuda")
    off = torch.empty(nq + 1, dtype=torch.int64, device="cuda")
    hits = torch.empty(40 * nq, dtype=torch.int32, device="cuda")

    def call():
        if how.startswith("knn"):
            return lib.lbvh_knn(tree.handle, q.data_ptr(), nq, k, idx.data_ptr(), d2.data_ptr(), None)
        return tree.query_into(q, lbvh.SPHERE, off, hits, radius=0.02)[0]

    assert lib.lbvh_test_hold_sort_tile(3) == lbvh.OK
    try:
        st = call()
        torch.cuda.synchronize()
    finally:
        assert lib.lbvh_test_hold_sort_tile(-1) == lbvh.OK
    assert st == lbvh.ERR_TIMEOUT
    assert bool((idx[nq:] == 7).all()) and bool((d2[nq:] == 7).all())
    tree.build(inputs.uniform_points(n, seed=3), lbvh.POINTS, 30)  # clears the flag
    assert call() == lbvh.OK
    few = 500  # few queries need no order
    if how.startswith("knn"):
        wi, wd = tree.knn(q[:few], k)
        assert torch.equal(idx[:few], wi) and torch.equal(d2[:few], wd)
    else:
        o, h = tree.query(q[:few], lbvh.SPHERE, radius=0.02)
        assert torch.equal(off[:few + 1], o) and torch.equal(hits[:h.numel()], h)
    tree.close()


def test_order_of_a_batch_that_gave_up():
    from paper_2402_00665_gb300 import lbvh
    lib = lbvh.load()
    sizes = [40_000, 30_000, 50_000]
    po = np.concatenate([[0], np.cumsum(sizes)]).astype(np.int64)
    pts = torch.from_numpy(inputs.uniform_points(int(po[-1]), seed=5)).cuda()
    q = torch.from_numpy(inputs.uniform_points(int(po[-1]), seed=6)).cuda()
    batch = lbvh.Batch()
    args = dict(queries=q, query_offsets=po, radius=0.02, capacity=60 * int(po[-1]))
    assert lib.lbvh_test_hold_sort_tile(3) == lbvh.OK
    try:
        st = batch.build_query(pts, po, lbvh.POINTS, 30, **args)[3]
        torch.cuda.synchronize()
    finally:
        assert lib.lbvh_test_hold_sort_tile(-1) == lbvh.OK
    assert st == lbvh.ERR_TIMEOUT
    fresh = lbvh.Batch()
    o, h, total, st = fresh.build_query(pts, po, lbvh.POINTS, 30, **args)
    assert st == lbvh.OK
    tree = lbvh.Tree().build(pts[:sizes[0]], lbvh.POINTS, 30)
    wo, wh = tree.query(q[:sizes[0]], lbvh.SPHERE, radius=0.02)
    assert torch.equal(o[:sizes[0] + 1], wo) and torch.equal(h[:wh.numel()], wh)
    for x in (batch, fresh, tree):
        x.close()
