"""Rays keep the order they are given in where 32 by 32 they lie together, and
are put in the order of cells where they do not: the same hits either way, for
rows and tiles of a camera, scattered rays, mixtures of both around the line
between them, and rays that hit nothing or are not finite."""
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


def camera(n):
    """float32[n, 8]: rays of a pinhole, in rows of 400."""
    i = np.arange(n)
    d = np.stack([(i % 400) / 400 - 0.5, (i // 400) / (n / 400) - 0.5, np.ones(n)], axis=1)
    out = np.zeros((n, 8), np.float32)
    out[:, :3] = [0.5, 0.5, -0.5]
    out[:, 4:7] = d / np.linalg.norm(d, axis=1, keepdims=True)
    out[:, 7] = np.inf
    return out


@pytest.mark.parametrize("kind", ["points", "boxes"])
@pytest.mark.parametrize("nq", [45_000, 120_003])  # 8 lanes per ray with an order, a thread per ray
@pytest.mark.parametrize("scattered", [0.0, 0.24, 0.26, 1.0])
def test_orders(kind, nq, scattered):
    from paper_2402_00665_gb300 import lbvh
    n = 20_000
    rng = np.random.default_rng(nq)
    c = inputs.uniform_points(n, seed=5)
    prims = c if kind == "points" else np.concatenate([c - 0.01, c + 0.01], axis=1).astype(np.float32)
    rays = camera(nq)
    runs = (nq + 31) // 32
    for r in rng.permutation(runs)[:int(scattered * runs)]:
        part = rays[32 * r:32 * r + 32]
        part[:, :3] = rng.random((len(part), 3))
        part[:, 4:7] = rng.standard_normal((len(part), 3))
        part[:, 7] = 0.3
    rays[11, 4] = np.nan
    rays[40, 3], rays[40, 7] = 1.0, 0.0
    rays[70, 4:7] = 0.0
    tree = lbvh.Tree().build(prims, lbvh.POINTS if kind == "points" else lbvh.BOXES, 63)
    q = torch.from_numpy(rays).cuda()
    off, hits = tree.query(q, lbvh.RAY)
    off, hits = off.cpu().numpy(), hits.cpu().numpy()
    for first in range(0, nq, 4000):  # too few for an order
        o, h = tree.query(q[first:first + 4000], lbvh.RAY)
        o, h = o.cpu().numpy(), h.cpu().numpy()
        assert np.array_equal(off[first:first + len(o)] - off[first], o)
        assert np.array_equal(hits[off[first]:off[first] + len(h)], h)
    tree.close()
