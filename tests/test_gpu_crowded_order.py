"""Queries that crowd into few cells of their order's grid (clusters far smaller
than the scene) are put in a finer order before they walk in packets: the same
hits and neighbours as by Algorithm 1, at the edges of the windows this is done
in, with queries outside the scene, and with a NaN and an infinity among them."""
from __future__ import annotations

import numpy as np
import pytest

from paper_2402_00665_gb300 import _build

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

NODES = 4  # walk variant: Algorithm 1, one thread per query
WINDOW = 4096


@pytest.fixture(scope="module", autouse=True)
def lib():
    if not torch.cuda.is_available():
        pytest.skip("needs a GPU")
    _build.build()
    from paper_2402_00665_gb300 import lbvh
    return lbvh.load()


def clusters(n, sigma, seed):
    """float32[n, 3]: 8 tight clusters in the unit cube and its two far corners; a NaN and an infinity in the queries'."""
    rng = np.random.default_rng(seed)
    centres = np.random.default_rng(99).random((8, 3))
    p = centres[rng.integers(0, 8, n)] + sigma * rng.standard_normal((n, 3))
    p[0], p[1] = 0.0, 1.0
    return p.astype(np.float32)


@pytest.mark.parametrize("kind", ["points", "boxes"])
@pytest.mark.parametrize("nq", [32 * WINDOW, 32 * WINDOW + 1, 33 * WINDOW - 1, 200_003])
@pytest.mark.parametrize("walk", [-1, 5])  # 5: as -1 with the queries ordered by 24 bits
def test_clusters(kind, nq, walk):
    from paper_2402_00665_gb300 import lbvh
    n, sigma = 150_000, 2e-4
    pts, q = clusters(n, sigma, 1), clusters(nq, sigma, 2)
    q[5, 1], q[6, 2] = np.nan, np.inf
    r = np.float32(0.08 * sigma)
    if kind == "boxes":
        pts, q = (np.concatenate([x - r, x + r], axis=1) for x in (pts, q))
    code, qkind = (lbvh.BOXES, lbvh.BOX) if kind == "boxes" else (lbvh.POINTS, lbvh.SPHERE)
    tree = lbvh.Tree().build(pts, code, 63)
    q = torch.from_numpy(q).cuda()
    radii = torch.full((nq,), float(r), device="cuda")
    radii[::3] *= 2.0
    kw = {} if kind == "boxes" else {"radii": radii}
    tree.set_tuning(-1, walk)
    got = [x.cpu() for x in tree.query(q, qkind, **kw)]
    tree.set_tuning(-1, NODES)
    want = [x.cpu() for x in tree.query(q, qkind, **kw)]
    assert torch.equal(got[0], want[0]) and torch.equal(got[1], want[1])
    if kind == "points" and walk == -1:  # 8 nearest neighbours, against the heap (as many as 40)
        idx, d2 = tree.knn(q, 8)
        widx, wd2 = tree.knn(q, 40)
        assert torch.equal(idx, widx[:, :8]) and torch.equal(d2, wd2[:, :8])
    tree.close()
