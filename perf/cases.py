"""The work a program has this library do, as cases that can be timed.

A case is a dict of plain values; ``prepare`` makes what the program holds
before the call, ``run`` makes the call through the public entry points of
the package and returns every output.  Fields and masks follow the recipes of
the workloads of this repository (sums of Gaussians, white noise, thresholded
sums, thinned Kuhn meshes), drawn on the GPU from the seed alone.
"""
from __future__ import annotations

import itertools
import math
import random

import torch

import paper_2409_03771_gb300 as msc

# The positive half of the 14-neighbour link, faces first.
LINK = [(1, 0, 0), (0, 1, 0), (0, 0, 1), (1, 1, 0), (1, 0, 1), (0, 1, 1), (1, 1, 1)]
MEMBERS = "bumps", "mixed"  # the fields of an ensemble or a request stream, in turn: computed and measured ones
CSR_PER_VERTEX = 13.7  # CSR entries per vertex of a Kuhn mesh with 40 % of its tetrahedra deleted


# ----------------------------------------------------------------------------
# cases


def listed():
    return [
        # the paper-shaped unit workload: one small field, segmented while an
        # interactive program waits; launches and latency are what it costs
        {"name": "segment-64", "kind": "segment", "nx": 64, "ny": 64, "nz": 64, "field": "mixed"},
        # an ordinary cropped volume: odd edges, rows that no vector access fits
        {"name": "segment-ragged", "kind": "segment", "nx": 181, "ny": 97, "nz": 131, "field": "mixed"},
        # a CT scan: 8-bit values held as float32, so nearly every vertex ties
        {"name": "segment-scan", "kind": "segment", "nx": 256, "ny": 256, "nz": 256, "field": "scan"},
        # a simulation field: few extrema, long steepest paths
        {"name": "segment-smooth-512", "kind": "segment", "nx": 512, "ny": 512, "nz": 512, "field": "smooth"},
        # the other end: millions of extrema and cells, short paths
        {"name": "segment-noise-512", "kind": "segment", "nx": 512, "ny": 512, "nz": 512, "field": "noise"},
        # features of a small odd volume, with the triangulation's neighbours
        {"name": "mask-ragged-14", "kind": "mask", "nx": 203, "ny": 150, "nz": 177, "conn": 14, "top": 0.5},
        # features of the largest volume, face neighbours
        {"name": "mask-1024-6", "kind": "mask", "nx": 1024, "ny": 1024, "nz": 1024, "conn": 6, "top": 0.1},
        # fragments of a damaged tetrahedral mesh
        {"name": "mesh-components", "kind": "mesh_cc", "edge": 256, "delete": 0.4},
        # the segmentation of a scalar field on a tetrahedral mesh, stage by
        # stage as the entry points for meshes have it
        {"name": "mesh-segment", "kind": "mesh_segment", "edge": 150, "delete": 0.1},
        # what follows a segmentation: which cells touch, and the arcs between
        # maxima with their saddles
        {"name": "graph-noise", "kind": "graph", "nx": 256, "ny": 256, "nz": 200, "field": "noise", "conn": 14,
         "sense": 1},
        # an ensemble of uneven grids, segmented again and again by one plan
        {"name": "batch-96", "kind": "batch", "count": 96, "low": 16, "high": 256, "dims_seed": 100},
        # a burst of requests of mixed kinds and sizes at a server
        {"name": "serve-12", "kind": "serve", "count": 12, "low": 32, "high": 256, "dims_seed": 7},
    ]


def _edges(rng, low, high, cap):
    """Three log-uniform edges whose product stays within cap."""
    e = [int(round(math.exp(rng.uniform(math.log(low), math.log(high))))) for _ in range(3)]
    while e[0] * e[1] * e[2] > cap:
        i = e.index(max(e))
        e[i] = max(1, e[i] // 2 + 1)
    return {"nx": e[0], "ny": e[1], "nz": e[2]}


def draw(rng):
    kind = rng.choice(["segment", "segment", "segment", "mask", "mask", "mesh_cc", "mesh_segment", "graph", "batch",
                       "serve"])
    if kind == "segment":
        return {"kind": kind, **_edges(rng, 24, 640, 1 << 27),
                "field": rng.choice(["bumps", "mixed", "scan", "smooth", "noise"])}
    if kind == "mask":
        return {"kind": kind, **_edges(rng, 48, 1024, 1 << 29), "conn": rng.choice([6, 14]),
                "top": rng.choice([0.1, 0.3, 0.5, 0.9])}
    if kind == "mesh_cc":
        return {"kind": kind, "edge": int(round(math.exp(rng.uniform(math.log(24), math.log(250))))),
                "delete": round(rng.uniform(0.1, 0.8), 2)}
    if kind == "mesh_segment":
        return {"kind": kind, "edge": int(round(math.exp(rng.uniform(math.log(24), math.log(190))))),
                "delete": round(rng.uniform(0.0, 0.5), 2)}
    if kind == "graph":
        return {"kind": kind, **_edges(rng, 32, 400, 1 << 24), "field": rng.choice(["mixed", "scan", "smooth", "noise"]),
                "conn": rng.choice([6, 14]), "sense": rng.choice([-1, 1])}
    if kind == "batch":
        return {"kind": kind, "count": int(round(math.exp(rng.uniform(math.log(8), math.log(128))))), "low": 16,
                "high": 220, "dims_seed": rng.randrange(1 << 20)}
    return {"kind": kind, "count": rng.randrange(3, 13), "low": 32, "high": 200, "dims_seed": rng.randrange(1 << 20)}


def _dims(case):
    return case["nx"], case["ny"], case["nz"]


def _batch_dims(case):
    r = random.Random(case["dims_seed"])
    lo, hi = math.log(case["low"]), math.log(case["high"])
    return [tuple(int(round(math.exp(r.uniform(lo, hi)))) for _ in range(3)) for _ in range(case["count"])]


def _serve_jobs(case):
    """(is a mask, cube edge) of each request: 30 % masks, edges log-uniform."""
    r = random.Random(case["dims_seed"])
    lo, hi = math.log(case["low"]), math.log(case["high"])
    return [(r.random() < 0.3, int(round(math.exp(r.uniform(lo, hi))))) for _ in range(case["count"])]


# ----------------------------------------------------------------------------
# inputs


def _generator(seed):
    return torch.Generator(device="cuda").manual_seed(seed)


def _gaussians(dims, count, low, high, gen, dtype=torch.float64):
    """sum_i A_i exp(-|p - c_i|^2 / (2 s_i^2)), A in [-1, 1], s = U[low, high] times the grid's mean edge."""
    nx, ny, nz = dims
    mean = (nx * ny * nz) ** (1.0 / 3.0)
    u = torch.rand((count, 5), generator=gen, device="cuda", dtype=torch.float64).tolist()
    axes = [torch.arange(k, dtype=torch.float64, device="cuda") for k in dims]
    acc = torch.zeros((nz, ny, nx), dtype=dtype, device="cuda")
    for cx, cy, cz, s, a in u:
        k = -0.5 / ((low + (high - low) * s) * mean) ** 2
        ex, ey, ez = (torch.exp(k * (ax - c * d) ** 2) for ax, c, d in zip(axes, (cx, cy, cz), dims))
        yz = ((2 * a - 1) * ez)[:, None] * ey[None, :]
        acc.addcmul_(yz[:, :, None].to(dtype), ex[None, None, :].to(dtype))
    return acc.reshape(-1)


def _field(dims, name, gen):
    n = dims[0] * dims[1] * dims[2]
    if name == "noise":  # uniform multiples of 2^-24
        return torch.rand(n, generator=gen, device="cuda", dtype=torch.float32)
    if name == "smooth":
        return _gaussians(dims, 64, 1 / 16, 3 / 16, gen).float()
    f = _gaussians(dims, 8, 1 / 16, 3 / 16, gen)
    if name == "bumps":
        return f.float()
    if name == "mixed":  # with a little noise
        return f.add_(torch.rand(n, generator=gen, device="cuda", dtype=torch.float32), alpha=1e-3).float()
    # scan: 8-bit values of the sum with measurement noise
    f.mul_(100.0).add_(torch.randn(n, generator=gen, device="cuda", dtype=torch.float32), alpha=3.0)
    return f.add_(100.0).round_().clamp_(0.0, 255.0).float()


def _mask(dims, top, gen):
    """uint8 mask of the top fraction of a sum of Gaussians' values (the threshold from a sample)."""
    f = _gaussians(dims, 64, 1 / 16, 3 / 16, gen, torch.float32)
    at = torch.randint(0, f.numel(), (min(f.numel(), 1 << 20),), generator=gen, device="cuda")
    return (f > torch.quantile(f[at], 1.0 - top)).to(torch.uint8)


def _mesh(edge, delete, gen):
    """int32 CSR of the edges of a Kuhn mesh on edge^3 vertices, a fraction of whose tetrahedra is deleted and
    whose vertex ids are permuted."""
    n = edge ** 3
    r = torch.arange(edge - 1, device="cuda", dtype=torch.int64)
    base = (r[None, None, :] + edge * (r[None, :, None] + edge * r[:, None, None])).reshape(-1)
    perm = torch.randperm(n, generator=gen, device="cuda")
    keys = []
    for p in itertools.permutations((1, edge, edge * edge)):
        b = base[torch.rand(base.numel(), generator=gen, device="cuda") >= delete]
        corner = [perm[b], perm[b + p[0]], perm[b + p[0] + p[1]], perm[b + sum(p)]]
        keys += [torch.minimum(u, v) * n + torch.maximum(u, v) for u, v in itertools.combinations(corner, 2)]
    und = torch.unique(torch.cat(keys))
    del keys
    both = torch.cat([und, und % n * n + und // n]).sort().values
    row = torch.zeros(n + 1, dtype=torch.int64, device="cuda")
    row[1:] = torch.cumsum(torch.bincount(both // n, minlength=n), 0)
    return row.int(), (both % n).int()


def _graph_input(case, seed):
    """Labels and order of a segmented field: order, maximum (minimum) labels, cell ids, cell count."""
    f = _field(_dims(case), case["field"], _generator(seed))
    order, asc, desc, ms, cells = _segment(f, _dims(case))
    return order, desc if case["sense"] > 0 else asc, ms, cells


def prepare(case, seed):
    gen = _generator(seed)
    kind = case["kind"]
    if kind == "segment":
        return {"case": case, "f": _field(_dims(case), case["field"], gen)}
    if kind == "mask":
        return {"case": case, "mask": _mask(_dims(case), case["top"], gen)}
    if kind in ("mesh_cc", "mesh_segment"):
        row, col = _mesh(case["edge"], case["delete"], gen)
        f = torch.rand(case["edge"] ** 3, generator=gen, device="cuda", dtype=torch.float32)
        return {"case": case, "row": row, "col": col, "f": f}
    if kind == "graph":
        order, label, ms, cells = (t.int() if torch.is_tensor(t) else t for t in _graph_input(case, seed))
        n = order.numel()
        arcs, pairs = n, 5 * n  # entries kept for the results; what a pass does not reach stays -1
        ws = max(msc.msc_workspace_bytes(op, n) for op in (msc.OP_EXTREMUM_GRAPH, msc.OP_ADJACENCY))
        return {"case": case, "order": order, "label": label, "ms": ms, "cells": cells,
                "arcs": [torch.full((arcs,), -1, dtype=torch.int32, device="cuda") for _ in range(3)],
                "pairs": [torch.full((pairs,), -1, dtype=torch.int32, device="cuda") for _ in range(2)],
                "count": torch.zeros(2, dtype=torch.int64, device="cuda"),
                "status": torch.zeros(2, dtype=torch.int32, device="cuda"),
                "ws": torch.empty(ws, dtype=torch.uint8, device="cuda")}
    if kind == "batch":
        b = msc.Batch(_batch_dims(case))
        for i, (d, part) in enumerate(zip(b.dims, b.split(b.f))):
            part.copy_(_field(d, MEMBERS[i % 2], gen))
        b.plan()
        return {"case": case, "batch": b}
    jobs = []
    for i, (is_mask, edge) in enumerate(_serve_jobs(case)):
        dims = (edge,) * 3
        jobs.append((is_mask, dims, _mask(dims, 0.3, gen) if is_mask else _field(dims, MEMBERS[i % 2], gen)))
    return {"case": case, "jobs": jobs, "server": msc.Server(16 << 30)}


# ----------------------------------------------------------------------------
# one pass


def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "segment":
        return msc.segment(state["f"], _dims(case))
    if kind == "mask":
        return msc.cc_mask(state["mask"], _dims(case), case["conn"])
    if kind == "mesh_cc":
        return msc.cc_mesh(state["row"], state["col"])
    if kind == "mesh_segment":
        order = msc.order(state["f"])
        asc, desc = msc.steepest_csr(order, state["row"], state["col"])
        asc, desc = msc.compress(asc, inplace=True), msc.compress(desc, inplace=True)
        return (order, asc, desc, *msc.ms_id(asc, desc))
    if kind == "graph":
        arcs, pairs, count, status, ws = (state[k] for k in ("arcs", "pairs", "count", "status", "ws"))
        n = state["order"].numel()
        codes = (msc.msc_extremum_graph(state["label"], state["order"], _dims(case), case["conn"], n, case["sense"],
                                        *arcs, arcs[0].numel(), count[:1], ws, ws.numel(), status[:1]),
                 msc.msc_adjacency_grid(state["ms"], _dims(case), case["conn"], state["cells"], *pairs,
                                        pairs[0].numel(), count[1:], ws, ws.numel(), status[1:]))
        if any(codes):
            raise RuntimeError(f"graph: {codes}")
        return [*arcs, *pairs, count, status]
    if kind == "batch":
        b = state["batch"]
        b.launch()
        return [b.order, b.asc, b.desc, b.ms, b.num_cells]
    srv = state["server"]
    tickets = [srv.submit_cc(t, dims, 6) if is_mask else srv.submit_segment(t, dims)
               for is_mask, dims, t in state["jobs"]]
    out = [srv.outputs(t) for t in tickets]
    for t in tickets:
        srv.release(t)
    return out


# ----------------------------------------------------------------------------
# the work that cannot be avoided


def work(case):
    """Inputs read once, outputs written once (graphs: the pairs of a typical field of the kind)."""
    kind = case["kind"]
    if kind in ("segment", "mask", "graph"):
        n = case["nx"] * case["ny"] * case["nz"]
        if kind == "segment":
            return {"bytes": 20 * n, "flops": 0}
        if kind == "mask":
            return {"bytes": 5 * n, "flops": 0}
        arcs, pairs = {"noise": (0.5, 2.5), "scan": (0.1, 0.3), "mixed": (0.05, 0.2), "smooth": (0, 0)}[case["field"]]
        return {"bytes": int(n * (12 + 12 * arcs + 8 * pairs)), "flops": 0}
    if kind in ("mesh_cc", "mesh_segment"):
        n = case["edge"] ** 3
        return {"bytes": int(n * (8 + 4 * CSR_PER_VERTEX + (16 if kind == "mesh_segment" else 0))), "flops": 0}
    if kind == "batch":
        return {"bytes": 20 * sum(x * y * z for x, y, z in _batch_dims(case)), "flops": 0}
    return {"bytes": sum((5 if is_mask else 20) * e ** 3 for is_mask, e in _serve_jobs(case)), "flops": 0}


# ----------------------------------------------------------------------------
# the same outputs from plain torch, in 64-bit integers


def _order(f):
    perm = torch.argsort(f.double() + 0.0, stable=True)
    order = torch.empty_like(perm)
    order[perm] = torch.arange(f.numel(), device=f.device)
    return order


def _shifted(dims, off):
    """Slices of a (nz, ny, nx) array holding the lower and the upper ends of the edges at a positive offset."""
    lo = tuple(slice(0, d - o) for d, o in zip(reversed(dims), reversed(off)))
    hi = tuple(slice(o, d) for d, o in zip(reversed(dims), reversed(off)))
    return lo, hi


def _roots(p):
    while True:
        q = p[p]
        if torch.equal(p, q):
            return p
        p = q


def _cells(asc, desc):
    keys, ms = torch.unique(asc * asc.numel() + desc, return_inverse=True)
    return ms, keys.numel()


def _segment(f, dims):
    order = _order(f)
    n = order.numel()
    at = order.view(dims[2], dims[1], dims[0])
    low, high = at.clone(), at.clone()
    for off in LINK:
        lo, hi = _shifted(dims, off)
        low[lo], low[hi] = torch.minimum(low[lo], at[hi]), torch.minimum(low[hi], at[lo])
        high[lo], high[hi] = torch.maximum(high[lo], at[hi]), torch.maximum(high[hi], at[lo])
    vertex = torch.empty_like(order)
    vertex[order] = torch.arange(n, device=order.device)
    asc = _roots(vertex[low.view(-1)])
    desc = _roots(vertex[high.view(-1)])
    return (order, asc, desc, *_cells(asc, desc))


def _components(n, edges, live=None):
    """Smallest vertex id of each component; `edges()` yields (lower ends, upper ends) id tensors."""
    lab = torch.arange(n, device="cuda")
    while True:
        before = lab
        lab = lab.clone()
        for u, v in edges():
            a, b = lab[u], lab[v]
            m = torch.minimum(a, b)
            lab.scatter_reduce_(0, a, m, "amin")
            lab.scatter_reduce_(0, b, m, "amin")
        lab = _roots(lab)
        if torch.equal(before, lab):
            return lab if live is None else torch.where(live, lab, -1)


def _mask_components(mask, dims, conn):
    live = (mask != 0).view(dims[2], dims[1], dims[0])
    ids = torch.arange(mask.numel(), device="cuda").view(live.shape)

    def edges():
        for off in LINK[:3 if conn == 6 else 7]:
            lo, hi = _shifted(dims, off)
            both = live[lo] & live[hi]
            yield ids[lo][both], ids[hi][both]

    return _components(mask.numel(), edges, mask != 0)


def _pairs(label, dims, conn, order=None, sense=1):
    """Distinct (smaller, larger) label pairs over the grid's edges, with each pair's crossing vertex at the
    highest (lowest) level when an order is given."""
    n = label.numel()
    lab = label.long().view(dims[2], dims[1], dims[0])
    level = None if order is None else order.long().view(lab.shape)
    keys, levels = [], []
    for off in LINK[:3 if conn == 6 else 7]:
        lo, hi = _shifted(dims, off)
        a, b = lab[lo], lab[hi]
        cross = a != b
        a, b = a[cross], b[cross]
        keys.append(torch.minimum(a, b) * n + torch.maximum(a, b))
        if level is not None:
            ends = level[lo][cross], level[hi][cross]
            levels.append(torch.minimum(*ends) if sense > 0 else torch.maximum(*ends))
    keys, inverse = torch.unique(torch.cat(keys), return_inverse=True)
    out = [keys // n, keys % n]
    if level is not None:
        best = torch.full((keys.numel(),), -1 if sense > 0 else n, device="cuda")
        best.scatter_reduce_(0, inverse, torch.cat(levels), "amax" if sense > 0 else "amin")
        vertex = torch.empty(n, dtype=torch.int64, device="cuda")
        vertex[order.long()] = torch.arange(n, device="cuda")
        out.append(vertex[best])
    return out


def exact(case, seed):
    kind = case["kind"]
    gen = _generator(seed)
    if kind == "segment":
        return _segment(_field(_dims(case), case["field"], gen), _dims(case))
    if kind == "mask":
        if case["nx"] * case["ny"] * case["nz"] > 1 << 27:
            return None
        return _mask_components(_mask(_dims(case), case["top"], gen), _dims(case), case["conn"])
    if kind in ("mesh_cc", "mesh_segment"):
        row, col = _mesh(case["edge"], case["delete"], gen)
        n = case["edge"] ** 3
        col = col.long()
        src = torch.repeat_interleave(torch.arange(n, device="cuda"), (row[1:] - row[:-1]).long())
        if kind == "mesh_cc":
            return _components(n, lambda: [(src, col)])
        order = _order(torch.rand(n, generator=gen, device="cuda", dtype=torch.float32))
        vertex = torch.empty_like(order)
        vertex[order] = torch.arange(n, device="cuda")
        asc = _roots(vertex[order.clone().scatter_reduce_(0, src, order[col], "amin")])
        desc = _roots(vertex[order.clone().scatter_reduce_(0, src, order[col], "amax")])
        return (order, asc, desc, *_cells(asc, desc))
    if kind == "graph":
        order, label, ms, _ = _graph_input(case, seed)
        arcs = _pairs(label, _dims(case), case["conn"], order, case["sense"])
        pairs = _pairs(ms, _dims(case), case["conn"])
        n = order.numel()
        out = [torch.nn.functional.pad(t[:size], (0, size - t[:size].numel()), value=-1)
               for t, size in [(t, n) for t in arcs] + [(t, 5 * n) for t in pairs]]
        return [*out, torch.tensor([arcs[0].numel(), pairs[0].numel()]), torch.zeros(2, dtype=torch.int64)]
    if kind == "batch":
        parts = [_segment(_field(d, MEMBERS[i % 2], gen), d) for i, d in enumerate(_batch_dims(case))]
        return [torch.cat([p[i] for p in parts]) for i in range(4)] + [torch.tensor([p[4] for p in parts])]
    out = []
    for i, (is_mask, edge) in enumerate(_serve_jobs(case)):
        dims = (edge,) * 3
        if is_mask:
            out.append({"label": _mask_components(_mask(dims, 0.3, gen), dims, 6)})
        else:
            order, asc, desc, ms, cells = _segment(_field(dims, MEMBERS[i % 2], gen), dims)
            out.append({"order": order, "asc": asc, "desc": desc, "ms": ms, "num_cells": cells})
    return out
