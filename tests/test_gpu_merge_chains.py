"""Clusters whose points come ever closer to their centre: their chains of leaves
leave more than the merges' lists hold, so in small builds elements wait where they
are for the last launch. Every field of the tree as the Karras build makes it, at
the sizes where the number of merges changes, and in no more than half as long
again as a build that climbs after its first merge."""
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


def clusters(n, decades, seed=0, count=64):
    """float32[n, 3]: `count` clusters, distances from their centres log-uniform over `decades`."""
    rng = np.random.default_rng(seed)
    d = rng.standard_normal((n, 3))
    d /= np.linalg.norm(d, axis=1, keepdims=True)
    r = 0.05 * 10.0 ** -rng.uniform(0.0, decades, (n, 1))
    return (rng.random((count, 3))[rng.integers(0, count, n)] + d * r).astype(np.float32)


def same(got, want):
    for k in want:
        a, b = np.asarray(got[k]), np.asarray(want[k])
        assert a.tobytes() == b.tobytes(), k


@pytest.mark.parametrize("bits", [30, 63])
@pytest.mark.parametrize("n", [257, 1023, 1025, 3000, 5119, 5121, 7000, 20_000, 24_575, 24_577])
def test_chains(n, bits):
    from paper_2402_00665_gb300 import lbvh
    for count, decades in ((64, 5.0), (3, 6.0)):
        pts = clusters(n, decades, seed=n, count=count)
        for kind, prims in ((lbvh.POINTS, pts), (lbvh.BOXES, np.concatenate([pts, pts + np.float32(1e-6)], axis=1))):
            want = lbvh.Tree().build(prims, kind, bits, algorithm=lbvh.BUILD_KARRAS)
            t = lbvh.Tree()
            for _ in range(2):  # the lists are left empty for the next build
                same(t.build(prims, kind, bits).export(), want.export())
            t.close()
            want.close()


def test_batch_of_chains():
    from paper_2402_00665_gb300 import lbvh
    parts = [clusters(n, 6.0, seed=n, count=c) for n, c in ((7000, 3), (1, 1), (300, 1), (9000, 40), (2000, 2))]
    off = np.concatenate([[0], np.cumsum([len(p) for p in parts])]).astype(np.int64)
    batch = lbvh.Batch()
    for _ in range(2):
        batch.build_query(torch.from_numpy(np.concatenate(parts)).cuda(), off, lbvh.POINTS, 63, capacity=1 << 22)
        for k, p in enumerate(parts):
            want = lbvh.Tree().build(p, lbvh.POINTS, 63, algorithm=lbvh.BUILD_KARRAS)
            same(batch.export(k), want.export())
            want.close()
    batch.close()


def construct_ms(pts):
    from paper_2402_00665_gb300 import lbvh
    t = lbvh.Tree()
    t.set_profiling(True)
    best = 1e9
    for _ in range(10):
        t.build(pts, lbvh.POINTS, 63)
        t.check()
        best = min(best, t.stage_times()["construct"])
    t.close()
    return best


def test_waiting_costs_no_more_than_climbing():
    """Where each merge waited for its own climbs, 20,000 points took twice as long as 33,000."""
    small, large = (torch.from_numpy(clusters(n, 5.0)).cuda() for n in (20_000, 33_000))
    assert construct_ms(small) < 1.5 * construct_ms(large)
