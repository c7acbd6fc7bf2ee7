"""Performance cases: the work that programs have this library do, through its
public entry points, from a thousand points (launches and latency) to 2^25
(throughput).

``listed()`` names the cases, ``draw(rng)`` gives others of the same ranges,
``prepare(case, seed)`` makes what a program has in hand before the call,
``run(state)`` is one pass, ``work(case)`` the bytes and operations a pass
cannot do without, ``exact(case, seed)`` the outputs in 64 bits where they are
computed numbers (the squared distances of k nearest neighbours; everything
else the library returns is whole numbers).

Inputs are synthetic like those of ``paper_2402_00665_gb300/inputs.py`` and of
the benchmark, drawn on the GPU: uniform points, points and boxes of a mixture
of 64 Gaussians, many clouds of log-uniform sizes, random ray segments; radii
hold 16 expected neighbours.
"""
from __future__ import annotations

import math
import random

import numpy as np
import torch

from paper_2402_00665_gb300 import lbvh

NEIGHBOURS = 16      # expected hits of a sphere query
COMPONENTS = 64      # Gaussians of a mixture,
SIGMA = 0.005        # their spread, and the
HALF = 1e-4          # median half extent of a mixture's boxes (2^25 of them; see _half)
RAY_TMAX = 0.05      # length of a ray segment
HITS_PER_QUERY = 32  # room for hits per query (the means are 9 to 21)


def listed() -> list:
    return [
        # the smallest call: one small cloud, built and queried with its own points; launches and
        # the host's part of the call are all of it
        {"name": "uniform_1000", "op": "build_query", "shape": "uniform", "n": 1000, "nq": 1000, "bits": 30, "self": True},
        # a small simulation's neighbour lists, rebuilt every step (the benchmark's small workload)
        {"name": "uniform_16384", "op": "build_query", "shape": "uniform", "n": 16384, "nq": 16384, "bits": 30,
         "self": True},
        # neighbour lists that the program reads on the host: the results go to page-locked memory
        {"name": "uniform_4m_to_host", "op": "to_host", "shape": "uniform", "n": 4_000_037, "nq": 4_000_037, "bits": 63},
        # the benchmark's default step: 2^25 points, 2^25 queries in a buffer of their own
        {"name": "uniform_2^25", "op": "build_query", "shape": "uniform", "n": 1 << 25, "nq": 1 << 25, "bits": 63,
         "self": False},
        # collision candidates: boxes against boxes on a clustered scene, at full size
        {"name": "boxes_2^25", "op": "build_query", "shape": "boxes", "n": 1 << 25, "nq": 1 << 24, "bits": 63,
         "self": False},
        # the same at an ordinary, odd size with short codes (many centres share a code)
        {"name": "boxes_3m_30bit", "op": "build_query", "shape": "boxes", "n": 3_000_017, "nq": 1_500_009, "bits": 30,
         "self": False},
        # k nearest neighbours of every point of a cloud (normals, k-NN graphs)
        {"name": "knn16_5m", "op": "knn", "shape": "uniform", "n": 5_000_011, "nq": 5_000_011, "bits": 63, "k": 16},
        # many independent clouds in one call, sizes log-uniform
        {"name": "batch_512_clouds", "op": "batch", "count": 512, "lo": 256, "hi": 262144, "bits": 30},
        # a step of a moving scene: new boxes on the kept topology, then some queries
        {"name": "refit_10m", "op": "refit", "shape": "uniform", "n": 10_000_019, "nq": 262_147, "bits": 63},
        # ray segments against a scene that stays
        {"name": "rays_1m_on_8m", "op": "resident", "shape": "boxes", "n": 1 << 23, "nq": 1 << 20, "bits": 63,
         "query": "ray"},
        # a few queries with radii of their own against a large clustered cloud that stays
        {"name": "probes_30k_on_8m", "op": "resident", "shape": "mixture", "n": 8_388_617, "nq": 30_011, "bits": 63,
         "query": "sphere"},
        # a burst of requests of mixed sizes, offered to the request server at once
        {"name": "served_31", "op": "served", "count": 31, "lo": 1024, "hi": 1 << 20, "bits": 30},
    ]


def _log_int(rng: random.Random, lo: int, hi: int) -> int:
    return int(math.exp(rng.uniform(math.log(lo), math.log(hi))))


def draw(rng: random.Random) -> dict:
    """One more case: an operation, then its size, spread over the logarithm of its range."""
    op = rng.choice(["build_query", "build_query", "build_query", "to_host", "knn", "batch", "refit", "resident",
                     "resident", "served"])
    bits = rng.choice([30, 63])
    if op in ("batch", "served"):
        hi = _log_int(rng, 16384, 262144) if op == "batch" else _log_int(rng, 131072, 1 << 20)
        count = _log_int(rng, 16, 512) if op == "batch" else rng.randint(4, 31)
        return {"op": op, "count": count, "lo": 256 if op == "batch" else 1024, "hi": hi, "bits": bits}
    top = {"build_query": 1 << 24, "to_host": 1 << 22, "knn": 1 << 22, "refit": 1 << 24, "resident": 1 << 23}[op]
    n = _log_int(rng, 1000, top) | 1
    shape = rng.choice(["uniform", "mixture"] if op in ("knn", "refit") else ["uniform", "mixture", "boxes"])
    case = {"op": op, "shape": shape, "n": n, "bits": bits}
    if op == "resident":
        case["nq"] = _log_int(rng, 1000, max(n // 2, 1001)) | 1
        case["query"] = rng.choice(["box", "ray"]) if shape == "boxes" else rng.choice(["sphere", "box"])
    elif op == "refit":
        case["nq"] = max(n // 38, 100)
    elif op == "build_query":
        case["self"] = rng.random() < 0.4
        case["nq"] = n if case["self"] else max(int(n * rng.uniform(0.3, 1.0)), 500)
    elif op == "knn":
        case["nq"] = n
        case["k"] = rng.choice([3, 8, 16, 32])
    else:
        case["nq"] = n
    return case


# ---------------------------------------------------------------- inputs

def _rng(seed: int, *parts: int) -> torch.Generator:
    mixed = np.random.SeedSequence([seed & 0xFFFFFFFF, *parts]).generate_state(1, np.uint64)[0]
    return torch.Generator(device="cuda").manual_seed(int(mixed) & 0x7FFFFFFFFFFFFFFF)


def _points(shape: str, n: int, seed: int, draw_no: int) -> torch.Tensor:
    """float32[n, 3]: uniform in [0, 1)^3, or of the seed's mixture."""
    g = _rng(seed, draw_no)
    if shape == "uniform":
        return torch.rand((n, 3), generator=g, device="cuda")
    centres = torch.rand((COMPONENTS, 3), generator=_rng(seed, 1000), device="cuda")
    p = torch.randn((n, 3), generator=g, device="cuda").mul_(SIGMA)
    return p.add_(centres[torch.randint(0, COMPONENTS, (n,), generator=g, device="cuda")])


def _half(case: dict) -> float:
    """Median half extent that keeps about as many boxes per query at every size: 9 per box query
    (extents follow the spacing), 16 per ray (the boxes' areas add up to the same)."""
    if case.get("query") == "ray":
        return HALF * math.sqrt((1 << 23) / case["n"])
    return HALF * ((1 << 25) / case["n"]) ** (1.0 / 3.0)


def _boxes(n: int, half: float, seed: int, draw_no: int) -> torch.Tensor:
    """float32[n, 6]: centres of the seed's mixture, lognormal half extents."""
    c = _points("mixture", n, seed, draw_no)
    h = torch.randn((n, 3), generator=_rng(seed, draw_no, 1), device="cuda").mul_(0.5).exp_().mul_(half)
    out = torch.empty((n, 6), device="cuda")
    torch.sub(c, h, out=out[:, :3])
    torch.add(c, h, out=out[:, 3:])
    return out


def _rays(n: int, seed: int, draw_no: int) -> torch.Tensor:
    """float32[n, 8]: origins at the mixture, directions uniform on the sphere, [0, RAY_TMAX]."""
    out = torch.zeros((n, 8), device="cuda")
    out[:, :3] = _points("mixture", n, seed, draw_no)
    d = torch.randn((n, 3), generator=_rng(seed, draw_no, 2), device="cuda")
    out[:, 4:7] = d / d.norm(dim=1, keepdim=True)
    out[:, 7] = RAY_TMAX
    return out


def _radius(shape: str, n: int) -> float:
    """The radius that holds NEIGHBOURS expected neighbours of a point."""
    density = float(n)
    if shape == "mixture":
        density = n / COMPONENTS / ((4.0 * math.pi) ** 1.5 * SIGMA ** 3)
    return float(np.float32((3.0 * NEIGHBOURS / (4.0 * math.pi * density)) ** (1.0 / 3.0)))


def _sizes(case: dict) -> list:
    """The instance sizes of a batch or a burst: part of the case, not of the seed."""
    r = random.Random(case["count"] * 1000003 + case["hi"])
    return [_log_int(r, case["lo"], case["hi"]) for _ in range(case["count"])]


def _queries(case: dict, seed: int) -> dict:
    """The query array, its kind and its radius for a case that queries one tree."""
    shape, n, nq = case["shape"], case["n"], case["nq"]
    kind = case.get("query", "box" if shape == "boxes" else "sphere")
    if kind == "ray":
        return {"queries": _rays(nq, seed, 20), "qkind": lbvh.RAY}
    if shape == "boxes":
        return {"queries": _boxes(nq, _half(case), seed, 20), "qkind": lbvh.BOX}
    q = _points(shape, nq, seed, 20)
    r = _radius(shape, n)
    if kind == "box":  # boxes of about the ball's volume
        return {"queries": torch.cat([q - 0.8 * r, q + 0.8 * r], dim=1), "qkind": lbvh.BOX}
    if case["op"] == "resident":  # every probe has a radius of its own
        radii = torch.rand((nq,), generator=_rng(seed, 21), device="cuda").add_(0.5).mul_(r)
        return {"queries": q, "qkind": lbvh.SPHERE, "radii": radii}
    return {"queries": q, "qkind": lbvh.SPHERE, "radius": r}


def prepare(case: dict, seed: int) -> dict:
    op, bits = case["op"], case["bits"]
    if op in ("batch", "served"):
        sizes = _sizes(case)
        off = np.concatenate([[0], np.cumsum(sizes)]).astype(np.int64)
        if op == "batch":
            pts = _points("uniform", int(off[-1]), seed, 1)
            radii = torch.from_numpy(np.repeat([_radius("uniform", k) for k in sizes], sizes).astype(np.float32)).cuda()
            return {"op": op, "batch": lbvh.Batch(), "prims": pts, "off": off, "radii": radii, "bits": bits,
                    "offsets": torch.empty(int(off[-1]) + 1, dtype=torch.int64, device="cuda"),
                    "hits": torch.zeros(HITS_PER_QUERY * int(off[-1]), dtype=torch.int32, device="cuda")}
        shapes = ["mixture" if k % 2 else "uniform" for k in range(len(sizes))]
        clouds = [_points(sh, m, seed, 100 + k) for k, (sh, m) in enumerate(zip(shapes, sizes))]
        return {"op": op, "server": lbvh.Server(48 << 30, slots=2, max_batch=256), "clouds": clouds, "bits": bits,
                "hits": [torch.zeros(HITS_PER_QUERY * m, dtype=torch.int32, device="cuda") for m in sizes],
                "radii": [_radius(sh, m) for sh, m in zip(shapes, sizes)]}
    shape, n, nq = case["shape"], case["n"], case["nq"]
    kind = lbvh.BOXES if shape == "boxes" else lbvh.POINTS
    prims = _boxes(n, _half(case), seed, 1) if shape == "boxes" else _points(shape, n, seed, 1)
    s = {"op": op, "tree": lbvh.Tree(), "prims": prims, "kind": kind, "bits": bits}
    if op == "knn":
        s["k"] = case["k"]
        return s
    s.update(_queries(case, seed))
    if case.get("self"):
        s["queries"] = prims
    if op == "to_host":
        s["offsets"] = torch.empty(nq + 1, dtype=torch.int64, pin_memory=True)
        s["hits"] = torch.zeros(HITS_PER_QUERY * nq, dtype=torch.int32, pin_memory=True)
    else:
        s["offsets"] = torch.empty(nq + 1, dtype=torch.int64, device="cuda")
        s["hits"] = torch.zeros(HITS_PER_QUERY * nq, dtype=torch.int32, device="cuda")
    if op in ("refit", "resident"):
        s["tree"].build(prims, kind, bits)
    if op == "refit":  # the scene a step later
        s["moved"] = prims + torch.randn(prims.shape, generator=_rng(seed, 30), device="cuda") * (0.3 * _radius(shape, n))
    return s


# ---------------------------------------------------------------- one pass

def _query(s: dict) -> list:
    """One query of the state's tree into the program's own arrays (the hits are the first offsets[nq] entries)."""
    call = s["tree"].query_into_host if s["op"] == "to_host" else s["tree"].query_into
    st, _ = call(s["queries"], s["qkind"], s["offsets"], s["hits"], radius=s.get("radius", 0.0), radii=s.get("radii"))
    if st != lbvh.OK:
        raise lbvh.LbvhError(st, "query")
    return [s["offsets"], s["hits"]]


def run(state: dict):
    s = state
    op = s["op"]
    if op == "batch":
        offsets, hits, _, st = s["batch"].build_query(s["prims"], s["off"], lbvh.POINTS, s["bits"], radii=s["radii"],
                                                      offsets=s["offsets"], hits=s["hits"])
        if st != lbvh.OK:
            raise lbvh.LbvhError(st, "batch")
        return [offsets, hits]
    if op == "served":
        tickets = [s["server"].submit(p, lbvh.POINTS, s["bits"], radius=r, capacity=HITS_PER_QUERY * p.shape[0])
                   for p, r in zip(s["clouds"], s["radii"])]
        out = []
        for t, mine in zip(tickets, s["hits"]):
            offsets, hits, info = s["server"].wait(t)
            if info["status"] != lbvh.OK:
                raise lbvh.LbvhError(info["status"], "served request")
            mine[:hits.numel()].copy_(hits)  # the program takes each answer into its own array
            out += [offsets, mine]
        return out
    if op == "refit":
        s["tree"].refit(s["moved"])
    elif op != "resident":
        s["tree"].build(s["prims"], s["kind"], s["bits"])
    if op == "knn":
        return list(s["tree"].knn(s["prims"], s["k"]))
    return _query(s)


# ---------------------------------------------------------------- what a pass cannot do without

def work(case: dict) -> dict:
    """Each input read once, each output written once; operations: a comparison per level of the sort
    and of the walk, and a distance or box test per result."""
    op = case["op"]
    if op in ("batch", "served"):
        n = nq = sum(_sizes(case))
        dim = qdim = 3
    else:
        n, nq = case["n"], case["nq"]
        dim = 6 if case["shape"] == "boxes" else 3
        qdim = {"ray": 8, "box": 6}.get(case.get("query"), dim)
    hits = 9.0 if dim == 6 else float(NEIGHBOURS)
    levels = math.log2(max(n, 2))
    if op == "knn":
        return {"bytes": 4 * dim * n + 8 * case["k"] * nq, "flops": n * levels + nq * (levels + 8 * case["k"])}
    b = 4 * qdim * nq + 8 * (nq + 1) + 4 * hits * nq
    f = nq * (levels + 8 * hits)
    if op == "resident":  # the tree's nodes on the queries' paths are read: their leaves at least
        return {"bytes": b + 16 * min(n, hits * nq), "flops": f}
    if op == "refit":  # order and codes in, boxes out
        return {"bytes": b + (4 * dim + 12 + 32 + 16) * n, "flops": f + 6 * n}
    return {"bytes": b + 4 * dim * n, "flops": f + n * levels}


# ---------------------------------------------------------------- 64-bit values

EXACT_PAIRS = 1 << 35  # most point-query pairs a brute force takes here


def exact(case: dict, seed: int):
    """Brute-force squared distances of the k nearest, in 64 bits; every other output is whole numbers."""
    if case["op"] != "knn" or case["n"] * case["nq"] > EXACT_PAIRS:
        return None
    p = _points(case["shape"], case["n"], seed, 1).double()
    rows, step = [], max(1, (1 << 27) // case["n"])
    for q in p.split(step):
        d2 = torch.zeros((q.shape[0], p.shape[0]), dtype=torch.float64, device=p.device)
        for a in range(3):
            d2 += (q[:, a, None] - p[None, :, a]).square_()
        rows.append(d2.topk(case["k"], dim=1, largest=False, sorted=True).values)
    return [None, torch.cat(rows)]
