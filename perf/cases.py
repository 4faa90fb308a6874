"""The work a program gives this library, as cases that can be timed and compared.

Every case is one call (or one round of calls) of the public Python interface
(paper_1409_8112_gb300.rtg), with inputs of the kinds the repository's benchmark and tests use:
roadmap builds from device or host points, batches of roadmaps, exact sets by brute force,
queries of new points against a stored index, and neighbour lists read from a stored roadmap.
Outputs are the whole CSR adjacency (row pointers and columns), in arrays of the program's own;
they are integers, so there is no rounding to allow for.

A program keeps one context for its life and builds one roadmap after another with it, on the
stream its other GPU work runs on; so does this file.
"""
import functools
import math

import numpy as np
import torch

from paper_1409_8112_gb300 import gen, rtg

_context = None


def _ctx():
    """The process's context: one for every case, as a program that builds many roadmaps has; it
    shares the program's torch stream."""
    global _context
    if _context is None:
        stream = torch.cuda.Stream()
        torch.cuda.set_stream(stream)
        _context = rtg.Context(0, stream=stream.cuda_stream)
    return _context


def listed():
    return [
        # the smallest call: a planner on the host builds one small 3-D roadmap and reads it
        # back; latency, launches and copies are all of it
        {"name": "small_host", "kind": "build", "n": 2000, "d": 3, "dtype": "f64", "m": 5,
         "r": 0.1, "cf": 1.0, "points": "uniform", "rotate": True, "symmetric": False,
         "host": True},
        # the benchmark's headline: one PRM*-style roadmap in a 6-D configuration space, points
        # already on the GPU
        {"name": "roadmap_100k", "kind": "build", "n": 100000, "d": 6, "dtype": "f64", "m": 8,
         "r": 0.0, "cf": 1.0, "points": "uniform", "rotate": True, "symmetric": False,
         "host": False},
        # a large roadmap in single precision
        {"name": "roadmap_1m", "kind": "build", "n": 1000000, "d": 6, "dtype": "f32", "m": 8,
         "r": 0.0, "cf": 1.0, "points": "uniform", "rotate": True, "symmetric": False,
         "host": False},
        # a ragged 9-D roadmap that stores every pair twice (for neighbour queries), from host
        # memory to pinned host memory
        {"name": "roadmap_9d_host_symmetric", "kind": "build", "n": 37777, "d": 9, "dtype": "f32",
         "m": 6, "r": 0.0, "cf": 1.0, "points": "uniform", "rotate": True, "symmetric": True,
         "host": True},
        # high recall with the paper's grids: shift-only, m = 20, cells of 1.35 r (Table II)
        {"name": "high_recall_shift_only", "kind": "build", "n": 100000, "d": 6, "dtype": "f64",
         "m": 20, "r": -1.0, "cf": 1.35, "points": "uniform", "rotate": False,
         "symmetric": False, "host": False},
        # clustered samples (narrow passages, informed sampling): dense cells and long rows
        {"name": "clustered_3d", "kind": "build", "n": 100000, "d": 3, "dtype": "f32", "m": 8,
         "r": 0.0, "cf": 1.0, "points": "clustered", "rotate": True, "symmetric": False,
         "host": False},
        {"name": "clustered_9d", "kind": "build", "n": 50000, "d": 9, "dtype": "f32", "m": 8,
         "r": 0.0, "cf": 1.0, "points": "clustered", "rotate": True, "symmetric": False,
         "host": False},
        # many roadmaps of mixed size and dimension in one call
        {"name": "batch_128", "kind": "batch", "count": 128, "nmin": 1000, "nmax": 200000,
         "dims": "3 6 9", "m": 6, "sizes": 1000},
        # the exact set, distances from tensor-core tiles
        {"name": "exact_tensor_200k", "kind": "brute", "n": 200000, "d": 6, "dtype": "f32",
         "tensor": "fp16"},
        # the exact set of a sample with the default arithmetic (the recall denominator)
        {"name": "exact_30k", "kind": "brute", "n": 30011, "d": 6, "dtype": "f64", "tensor": ""},
        # new points looked up in the stored grids of a roadmap (a planner's query phase)
        {"name": "query_new_points", "kind": "query", "n": 100000, "nq": 100000, "d": 6,
         "dtype": "f64", "m": 8},
        # the neighbour lists of a subset of a stored roadmap's points
        {"name": "neighbour_lists", "kind": "neighbours", "n": 100000, "nq": 10000, "d": 6,
         "dtype": "f64", "m": 8},
    ]


def _log_int(rng, lo, hi):
    return int(math.exp(rng.uniform(math.log(lo), math.log(hi + 1))))


def draw(rng):
    kind = rng.choice(["build", "build", "build", "high_recall", "clustered", "batch", "brute",
                       "brute", "query", "neighbours"])
    if kind == "build":
        n, m = _log_int(rng, 1000, 1000000), rng.randint(4, 10)
        n = min(n, 8000000 // m)
        return {"kind": "build", "n": n, "d": rng.randint(2, 9), "dtype": rng.choice(["f32", "f64"]),
                "m": m, "r": 0.0, "cf": rng.choice([1.0, 1.0, 1.1]), "points": "uniform",
                "rotate": True, "symmetric": rng.random() < 0.3, "host": rng.random() < 0.3}
    if kind == "high_recall":
        return {"kind": "build", "n": _log_int(rng, 3000, 100000), "d": rng.choice([3, 6]),
                "dtype": "f64", "m": rng.randint(12, 24), "r": -1.0,
                "cf": round(rng.uniform(1.1, 1.35), 3), "points": "uniform",
                "rotate": rng.random() < 0.5, "symmetric": False, "host": False}
    if kind == "clustered":
        return {"kind": "build", "n": _log_int(rng, 5000, 50000), "d": rng.randint(3, 9),
                "dtype": "f32", "m": rng.randint(5, 8), "r": 0.0, "cf": 1.0,
                "points": "clustered", "rotate": True, "symmetric": False, "host": False}
    if kind == "batch":
        return {"kind": "batch", "count": rng.randint(4, 100), "nmin": 500,
                "nmax": _log_int(rng, 5000, 150000), "dims": rng.choice(["3 6 9", "2 3", "6", "4 7"]),
                "m": rng.randint(4, 6), "sizes": rng.randint(0, 10 ** 6)}
    if kind == "brute":
        tensor = rng.choice(["", "fp16", "bf16"])
        return {"kind": "brute", "n": _log_int(rng, 1500, 150000 if tensor else 40000),
                "d": rng.randint(2, 12), "dtype": rng.choice(["f32", "f64"]), "tensor": tensor}
    return {"kind": kind, "n": _log_int(rng, 5000, 100000), "nq": _log_int(rng, 500, 100000),
            "d": rng.randint(3, 8), "dtype": rng.choice(["f32", "f64"]), "m": rng.randint(5, 10)}


def _np_dtype(name):
    return np.float64 if name == "f64" else np.float32


def _radius(case):
    """0: expected degree 2 ln n at uniform density; -1: the radius of Eq. 2; else as given."""
    if case["r"] == 0.0:
        return gen.radius_for_degree(case["n"], case["d"])
    if case["r"] < 0.0:
        return gen.radius_fmt(case["n"], case["d"])
    return case["r"]


def _points(kind, seed, n, d, dtype):
    if kind == "clustered":  # 8 Gaussians of sigma 0.05, clipped to the unit cube
        return gen.points_mixture(seed, n, d, k=8, sigma=0.05, dtype=dtype)
    return gen.points_uniform(seed, n, d, dtype)


def _roadmaps(case):
    """(n, d) of every roadmap of a batch: fixed by the case."""
    g = np.random.default_rng(case["sizes"])
    n = gen.log_uniform_int(g, case["nmin"], case["nmax"], case["count"])
    d = g.choice([int(x) for x in case["dims"].split()], case["count"])
    return [(int(a), int(b)) for a, b in zip(n, d)]


def prepare(case, seed):
    ctx = _ctx()
    kind = case["kind"]
    shapes = _shapes(case)
    if kind == "build":
        n, d, m, r = case["n"], case["d"], case["m"], _radius(case)
        pts = _points(case["points"], seed, n, d, _np_dtype(case["dtype"]))
        T = gen.transforms(seed, d, m, case["cf"] * r, 0 if case["rotate"] else gen.SHIFT_ONLY)
        s = {"case": case, "r": r, "c": case["cf"] * r, "T": T}
        if case["host"]:  # pinned, as a program that cares for its transfers has them
            s["points"] = torch.from_numpy(pts).pin_memory().numpy()
            s["room"] = tuple(torch.zeros(k, dtype=t, pin_memory=True).numpy() for k, t in
                              ((shapes[0][0] + 1, torch.int64), (shapes[0][1], torch.int32)))
        else:
            s["points"] = torch.from_numpy(pts).cuda()
            s["room"] = _room(shapes[0])
        return s
    if kind == "batch":
        items = []
        for k, (n, d) in enumerate(_roadmaps(case)):
            r = gen.radius_for_degree(n, d)
            one = seed * 1000 + k
            items.append((torch.from_numpy(gen.points_uniform(one, n, d, np.float32)).cuda(), r,
                          gen.transforms(one, d, case["m"], r), r))
        return {"case": case, "items": items,
                "room": _room((sum(x[0] for x in shapes), sum(x[1] for x in shapes)))}
    n, d, dtype = case["n"], case["d"], _np_dtype(case["dtype"])
    r = gen.radius_for_degree(n, d)
    pts = torch.from_numpy(gen.points_uniform(seed, n, d, dtype)).cuda()
    if kind == "brute":
        return {"case": case, "points": pts, "r": r, "room": _room(shapes[0])}
    T = gen.transforms(seed, d, case["m"], r)
    if kind == "neighbours":
        graph = ctx.all_pairs(pts, r, T, r, symmetric=True)
        which = np.random.default_rng(seed).integers(0, n, case["nq"], dtype=np.int32)
        return {"case": case, "graph": graph, "queries": torch.from_numpy(which).cuda(),
                "room": _room(shapes[0])}
    index = ctx.index(pts, r, T, r)
    new = torch.from_numpy(gen.points_uniform(seed + 500009, case["nq"], d, dtype)).cuda()
    return {"case": case, "index": index, "queries": new, "room": _room(shapes[0])}


class _DeviceArray:
    """A part of a result's device memory, for torch to copy from."""

    def __init__(self, ptr, count, typestr):
        self.__cuda_array_interface__ = {"shape": (count,), "typestr": typestr,
                                         "data": (ptr, False), "version": 2}


def _room(shape):
    """The program's own device arrays for a CSR of (rows, entries) of at most that size."""
    return (torch.zeros(shape[0] + 1, dtype=torch.int64, device="cuda"),
            torch.zeros(shape[1], dtype=torch.int32, device="cuda"))


def _keep(result, room):
    """Copies a result into the program's arrays (same stream) and gives it back."""
    rows, cols = room
    if result.nnz > cols.numel():
        raise RuntimeError("the program's arrays are too small for this result")
    rows.copy_(torch.as_tensor(_DeviceArray(result.csr.row_ptr, result.n + 1, "<i8"),
                               device="cuda"))
    if result.nnz:
        cols[:result.nnz].copy_(torch.as_tensor(
            _DeviceArray(result.csr.col, result.nnz, "<i4"), device="cuda"))
    result.release()
    return room


def run(state):
    case, ctx = state["case"], _ctx()
    kind = case["kind"]
    if kind == "build":
        res = ctx.all_pairs(state["points"], state["r"], state["T"], state["c"],
                            symmetric=case["symmetric"])
        if not case["host"]:
            return _keep(res, state["room"])
        res.download(state["room"])
        res.release()
        return state["room"]
    if kind == "batch":
        res, offsets = ctx.batch_all_pairs(state["items"], case["m"])
        return (*_keep(res, state["room"]), offsets)
    if kind == "brute":
        res = ctx.brute_force(state["points"], state["r"], tensor=case["tensor"] or None)
    elif kind == "query":
        res = state["index"].query(state["queries"])
    else:
        res = ctx.query_neighbors(state["graph"], state["queries"])
    return _keep(res, state["room"])


# ---- what a pass cannot do without ----------------------------------------------------------

@functools.lru_cache(maxsize=None)
def _pair_share(points, n, d, r, c, m, rotate, most):
    """Share of all point pairs that lie within r, and that also share a cell of one of m grids,
    from a sample of points of the same distribution."""
    k = min(n, most)
    p = _points(points, 1, k, d, np.float64)
    T = gen.transforms(1, d, m, c, 0 if rotate else gen.SHIFT_ONLY)
    sq = (p * p).sum(1)
    near = np.triu((sq[:, None] + sq[None, :] - 2.0 * (p @ p.T)) <= r * r, 1)
    i, j = np.nonzero(near)
    found = np.zeros(len(i), dtype=bool)
    for t in range(m):
        R, s = T[t, :d * d].reshape(d, d), T[t, d * d:]
        cell = np.floor((p @ R.T + s) / c)
        found |= (cell[i] == cell[j]).all(1)
    pairs = k * (k - 1) / 2
    return len(i) / pairs, float(found.sum()) / pairs


def _parts(case):
    """The parts of a pass, each as (points or queries n, d, coordinate bytes, reported entries,
    grid lookups): one, or one per roadmap."""
    kind = case["kind"]
    if kind == "batch":
        out = []
        for n, d in _roadmaps(case):
            r = gen.radius_for_degree(n, d)
            found = _pair_share("uniform", n, d, r, r, case["m"], True, 700)[1] * n * (n - 1) / 2
            out.append((n, d, 4, found, n * case["m"]))
        return out
    n, d, esz = case["n"], case["d"], 8 if case["dtype"] == "f64" else 4
    if kind == "build":
        r, m = _radius(case), case["m"]
        share = _pair_share(case["points"], n, d, r, case["cf"] * r, m, case["rotate"], 3000)[1]
        return [(n, d, esz, share * n * (n - 1) / 2 * (2 if case["symmetric"] else 1), n * m)]
    r = gen.radius_for_degree(n, d)
    if kind == "brute":
        share = _pair_share("uniform", n, d, r, r, 1, True, 3000)[0]
        return [(n, d, esz, share * n * (n - 1) / 2, 0)]
    share = _pair_share("uniform", n, d, r, r, case["m"], True, 3000)[1]
    if kind == "neighbours":  # an index and two row pointers in, a row pointer and the list out
        return [(case["nq"], 0, 0, share * n * case["nq"], 0)]
    return [(case["nq"], d, esz, share * n * case["nq"], case["nq"] * case["m"])]


def _shapes(case):
    """(rows, entries) a program makes room for: three times the entries it expects, and some."""
    return [(n, int(3.0 * found) + 40 * n + 4096) for n, _, _, found, _ in _parts(case)]


def work(case):
    """Points (and transforms) in, row pointers and columns out; the rotations of every point or
    query, and one distance per reported entry (per pair for an exact set)."""
    total = {"bytes": 0.0, "flops": 0.0}
    for n, d, esz, found, lookups in _parts(case):
        total["bytes"] += n * d * esz + 8 * (n + 1) + 4 * found
        if lookups:
            total["bytes"] += 8 * (d * d + d) * (lookups // n)
            total["flops"] += 2.0 * lookups * d * d + 3.0 * d * found
        else:
            total["flops"] += 3.0 * d * n * (n - 1) / 2
    if case["kind"] == "neighbours":
        total["bytes"] += 20 * case["nq"] + 4 * found
    if case["kind"] == "query":
        total["bytes"] += case["n"] * case["d"] * (8 if case["dtype"] == "f64" else 4)
    return total
