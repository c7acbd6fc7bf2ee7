"""The pool for hits past a query's slot: a small share of the walk's scratch,
so that trees queried once hold little, and larger after a query that ran out
of it; the lists are the same either way."""
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


@pytest.mark.parametrize("nq", [64, 1024, 4096, 20_000])
def test_a_small_tree_queried_once_holds_little(nq):
    from paper_2402_00665_gb300 import lbvh
    n = 1000
    t = lbvh.Tree().build(inputs.uniform_points(n, seed=1), lbvh.POINTS, 30)
    before = t.device_bytes()
    t.query(inputs.uniform_points(nq, seed=2), lbvh.SPHERE, radius=0.05)
    # per query: 256 bytes of slots, 32 of the pool (at least 256 KB), 12 of counts and lists, 24 of the
    # order's keys and 1 of look-back words; the leaf blocks and rounding: 128 KB
    assert t.device_bytes() - before <= 325 * nq + (256 << 10) + (128 << 10)
    t.close()


def test_the_pool_grows_after_it_ran_out():
    from paper_2402_00665_gb300 import lbvh
    n, nq = 4000, 2000
    pts, q = inputs.uniform_points(n, seed=3), inputs.uniform_points(nq, seed=4)
    want = lbvh.Tree().build(pts, lbvh.POINTS, 63)
    want.set_tuning(-1, NODES)
    off, hits = want.query(q, lbvh.SPHERE, radius=0.4)
    chunks = int(((off.diff() - 64).clamp(min=0) + 62).div(63, rounding_mode="floor").sum())
    assert 4 * 1024 < chunks < 65536  # the first pool has 1,024
    t = lbvh.Tree().build(pts, lbvh.POINTS, 63)
    held = []
    for _ in range(8):
        o, h = t.query(q, lbvh.SPHERE, radius=0.4)
        assert torch.equal(o, off) and torch.equal(h, hits)
        held.append(t.device_bytes())
    assert held[1] > held[0] and held[-1] == held[-2]
    assert held[-1] - held[0] <= 16 << 20
    t.close()
    want.close()
