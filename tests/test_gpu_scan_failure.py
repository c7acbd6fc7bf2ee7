"""The scan of a query's counts when one of its waits runs out, without a fault:
a tile that publishes nothing (lbvh_test_hold_scan_tile) makes the later tiles'
bounded look-back waits end after about a second. Batches enqueue the copies
behind the scan without asking the host, with offsets that no longer add up to
the total: no hit may be written, and the call reports LBVH_ERR_TIMEOUT."""
from __future__ import annotations

import numpy as np
import pytest

from paper_2402_00665_gb300 import _build, inputs

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

TILE = 4096


@pytest.fixture(scope="module", autouse=True)
def lib():
    if not torch.cuda.is_available():
        pytest.skip("needs a GPU")
    _build.build()
    from paper_2402_00665_gb300 import lbvh
    return lbvh.load()


def scene(long_lists: bool):
    """300 points, four tiles of queries: many hits in the first two tiles, few in the last two; with
    `long_lists` the first tiles' lists run past a query's slot (64 hits)."""
    pts = inputs.uniform_points(300, seed=1)
    q = inputs.uniform_points(4 * TILE, seed=2)
    radii = np.full(4 * TILE, 0.45 if long_lists else 0.25, np.float32)
    radii[2 * TILE:] = 0.05
    return torch.from_numpy(pts).cuda(), torch.from_numpy(q).cuda(), torch.from_numpy(radii).cuda()


@pytest.mark.parametrize("long_lists", [False, True])
def test_batch_writes_nothing_and_the_next_one_recovers(lib, long_lists):
    from paper_2402_00665_gb300 import lbvh
    pts, q, radii = scene(long_lists)
    po, qo = np.array([0, 300], np.int64), np.array([0, 4 * TILE], np.int64)
    tree = lbvh.Tree().build(pts, lbvh.POINTS, 30)
    want_off, want_hits = tree.query(q, lbvh.SPHERE, radii=radii)
    assert bool((want_off.diff()[:2 * TILE] > 64).any()) == long_lists
    # room for the last two tiles' lists, which is the total when tile 1 publishes nothing, in a larger buffer
    cap = int(want_off[-1] - want_off[2 * TILE])
    room = torch.full((want_hits.numel() + 64,), -7, dtype=torch.int32, device="cuda")
    assert cap < int(want_off[TILE])
    batch = lbvh.Batch()
    assert lib.lbvh_test_hold_scan_tile(1) == lbvh.OK
    try:
        _, _, _, st = batch.build_query(pts, po, lbvh.POINTS, 30, q, qo, radii=radii, hits=room[:cap], capacity=cap)
    finally:
        assert lib.lbvh_test_hold_scan_tile(-1) == lbvh.OK
    assert st == lbvh.ERR_TIMEOUT
    assert bool((room == -7).all())
    batch.close()
    batch = lbvh.Batch()
    off, hits, total, st = batch.build_query(pts, po, lbvh.POINTS, 30, q, qo, radii=radii, hits=room)
    assert st == lbvh.OK and total == want_hits.numel()
    assert torch.equal(off, want_off) and torch.equal(room[:total], want_hits)
    batch.close()
    tree.close()


def test_query_reports_the_wait_and_the_next_one_recovers(lib):
    from paper_2402_00665_gb300 import lbvh
    pts, q, radii = scene(False)
    tree = lbvh.Tree().build(pts, lbvh.POINTS, 30)
    want_off, want_hits = tree.query(q, lbvh.SPHERE, radii=radii)
    off = torch.empty(4 * TILE + 1, dtype=torch.int64, device="cuda")
    hits = torch.full((want_hits.numel(),), -7, dtype=torch.int32, device="cuda")
    assert lib.lbvh_test_hold_scan_tile(2) == lbvh.OK
    try:
        st, _ = tree.query_into(q, lbvh.SPHERE, off, hits, radii=radii)
    finally:
        assert lib.lbvh_test_hold_scan_tile(-1) == lbvh.OK
    assert st == lbvh.ERR_TIMEOUT and bool((hits == -7).all())
    st, total = tree.query_into(q, lbvh.SPHERE, off, hits, radii=radii)
    assert st == lbvh.OK and total == want_hits.numel()
    assert torch.equal(off, want_off) and torch.equal(hits, want_hits)
    tree.close()


def test_hook_argument_checked(lib):
    from paper_2402_00665_gb300 import lbvh
    assert lib.lbvh_test_hold_scan_tile(-2) == lbvh.ERR_INVALID
