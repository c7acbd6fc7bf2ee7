"""Queries that cannot have the scratch of the walks over leaf blocks (the
library's allocations above a limit fail) answer by the walks that need none,
with the same results, and take the others again once there is room."""
from __future__ import annotations

import contextlib

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


@contextlib.contextmanager
def limit(lib, max_bytes):
    assert lib.lbvh_test_limit_allocation(max_bytes) == 0
    try:
        yield
    finally:
        assert lib.lbvh_test_limit_allocation(0) == 0


def points(n, seed):
    return torch.from_numpy(inputs.uniform_points(n, seed=seed)).cuda()


@pytest.mark.parametrize("k,nq,slots,wants", [(16, 20_000, 20_000 * 512, True), (32, 20_000, 20_000 * 1024, True),
                                              (32, 12_000, 12_000 * 1024, False),  # below a query per 4 leaves: the heap
                                              (8, 300, None, True), (3, 300, None, True)])
def test_knn(lib, k, nq, slots, wants):
    """Packets without their slots, and 8 lanes per query without the leaf blocks."""
    from paper_2402_00665_gb300 import lbvh
    n = 60_000 if slots else 200_000
    p, q = points(n, 1), points(nq, 2)
    want = lbvh.Tree().build(p, lbvh.POINTS, 63)
    idx, d2 = want.knn(q, k)
    t = lbvh.Tree().build(p, lbvh.POINTS, 63)
    with limit(lib, slots - 1 if slots else 4 * n):  # the blocks of n leaves take 4.6 n
        for _ in range(2):
            i, d = t.knn(q, k)
            assert torch.equal(i, idx) and torch.equal(d, d2)
    held = t.device_bytes()
    i, d = t.knn(q, k)
    assert torch.equal(i, idx) and torch.equal(d, d2)
    assert (t.device_bytes() > held) == wants  # the scratch was had this time
    t.close()
    want.close()


@pytest.mark.parametrize("nq", [500, 2500])  # in input order, and enough for an order
def test_range(lib, nq):
    """8 lanes per query without the leaf blocks."""
    from paper_2402_00665_gb300 import lbvh
    n = 400_000
    p, q = points(n, 3), points(nq, 4)
    r = float(inputs.radius_for_neighbours(n))
    want = lbvh.Tree().build(p, lbvh.POINTS, 63)
    off, hits = want.query(q, lbvh.SPHERE, radius=r)
    t = lbvh.Tree().build(p, lbvh.POINTS, 63)
    with limit(lib, 4 * n):
        o, h = t.query(q, lbvh.SPHERE, radius=r)
        assert torch.equal(o, off) and torch.equal(h, hits)
    held = t.device_bytes()
    o, h = t.query(q, lbvh.SPHERE, radius=r)
    assert torch.equal(o, off) and torch.equal(h, hits)
    assert t.device_bytes() > held
    t.close()
    want.close()


def test_packets(lib):
    """The other buffers are there from a walk of the nodes; the leaf blocks are not."""
    from paper_2402_00665_gb300 import lbvh
    n = nq = 120_001
    p, q = points(n, 5), points(nq, 6)
    r = float(inputs.radius_for_neighbours(n))
    t = lbvh.Tree().build(p, lbvh.POINTS, 30)
    t.set_tuning(-1, 4)  # Algorithm 1, one thread per query
    off, hits = t.query(q, lbvh.SPHERE, radius=r)
    t.set_tuning(-1, -1)
    held = t.device_bytes()
    for room in (4 * n, 0):
        with limit(lib, room):
            o, h = t.query(q, lbvh.SPHERE, radius=r)
            assert torch.equal(o, off) and torch.equal(h, hits)
        assert (t.device_bytes() > held + 4 * n) == (room == 0)
    t.close()
