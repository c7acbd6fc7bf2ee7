"""What a server's admission counts for a request covers every device buffer
that grows with it (no GPU needed: sizes alone decide)."""
from __future__ import annotations

import ctypes

import pytest

from paper_2402_00665_gb300 import _build, lbvh


def spill_bytes(nq: int) -> int:
    """The pool for hits past a query's slot: chunks of 64 words, an eighth of nq up to 65,536, a sixteenth beyond."""
    return 256 * max(min(nq // 8, 65536), nq // 16)


def pack_bytes(n: int) -> int:
    """Boxes of blocks of 8 leaves, of 8 blocks and so on, heights padded to 8."""
    total, blocks = 0, n
    while blocks > 1 or total == 0:
        blocks = -(-blocks // 8)
        total += blocks
    return 32 * total


def pend_bytes(n: int) -> int:
    """Lists of 32 elements (16 bytes each) per group of 128 leaves, and above them per 8 groups, 5, 5, ..."""
    lists = -(-n // 128)
    total, each = lists, 8
    while lists > 1:
        lists = -(-lists // each)
        total, each = total + lists, 5
    return 512 * total


@pytest.mark.parametrize("kind,qkind", [(0, 0), (0, 1), (1, 0), (1, 1)])
@pytest.mark.parametrize("n,nq", [(1, 1), (100, 1000), (1000, 4096), (20_000, 20_000), (1_000_000, 70_000),
                                  (3_000_001, 2_000_003), (1 << 25, 1 << 25)])
def test_estimate_covers_the_buffers(n, nq, kind, qkind):
    lib = lbvh.load(_build.build())
    capacity = 32 * nq
    req = lbvh._Request(None, n, kind, 30, None, nq, qkind, 0.1, None, None, None, capacity, 0)
    got = lib.lbvh_request_bytes(ctypes.byref(req))
    prim, qsz = (12, 24)[kind], (12, 24)[qkind]
    tree = n * (prim + 2 * 8 + 2 * 4 + 32 + (16, 32)[kind] + 8) + pack_bytes(n) + pend_bytes(n)
    walk = nq * (qsz + 4 + 8 + 4 + 256 + 4 + 4 + 2 * 8 + 2 * 4) + nq // 4 + spill_bytes(nq)
    out = 8 * nq + 4 * capacity
    assert got >= tree + walk + out
    assert got <= 1.5 * (tree + walk + out)
    req.nq = -1
    assert lib.lbvh_request_bytes(ctypes.byref(req)) == 0
    assert lib.lbvh_request_bytes(None) == 0
