"""Performance cases of the coloring library: whole calls through the Python entry points.

A case colors (or orders) graphs of one kind and size; the graph's edges and the priority seed come
from the seed, its sizes from the case alone.  Graphs are made on the GPU:

  er        G(n, M), M = n * degree / 2 uniform pairs, symmetrised, deduplicated
  rmat      R-MAT (a, b, c, d = .57, .19, .19, .05), edge factor `ef`, ids permuted at random; n need
            not be a power of two (edges that touch an id past n are dropped)
  stencil   27-point stencil on an nx x ny x nz grid, natural ids
  grid      5-point stencil on an nx x ny grid, natural ids

Left out: the in-place mode, whose colors differ from run to run by design (it reads colors while
other threads write them), so that two runs cannot be compared value by value.
"""
import math
import random

import numpy as np
import torch

import paper_1509_08267_gb300 as gc

DEV = "cuda"


def listed():
    return [
        # one small interactive call (a task graph, a register-interference graph): latency only
        {"name": "er-1k-det", "op": "color", "graph": "er", "n": 1000, "degree": 8.0},
        # the repository's small configuration: G(10,000, degree 16)
        {"name": "er-10k-det", "op": "color", "graph": "er", "n": 10000, "degree": 16.0},
        # a mid-size social / web graph with an odd vertex count, colored one at a time
        {"name": "rmat-150k-det", "op": "color", "graph": "rmat", "n": 150001, "ef": 16},
        # a large graph without hubs (sparse-matrix coloring): every row is short
        {"name": "er-1m-det", "op": "color", "graph": "er", "n": 1000003, "degree": 32.0},
        # the repository's mesh configuration: finite-element / structured-grid coloring
        {"name": "stencil-256-det", "op": "color", "graph": "stencil", "nx": 256, "ny": 256, "nz": 256},
        # the repository's headline configuration: R-MAT scale 22
        {"name": "rmat-4m-det", "op": "color", "graph": "rmat", "n": 1 << 22, "ef": 16},
        # a caller whose arrays live in (pinned) host memory: copies in and out are part of the call
        {"name": "rmat-1m-host-det", "op": "color", "graph": "rmat", "n": 1 << 20, "ef": 16, "home": "host"},
        # fewest colors: sequential First Fit order under the smallest-last key (peeling + ordered rounds)
        {"name": "rmat-500k-ordered-sl", "op": "color", "graph": "rmat", "n": 500000, "ef": 16, "mode": "ordered",
         "priority": gc.PRIORITY_SMALLEST_LAST},
        # one recoloring pass over a coloring the caller already has
        {"name": "rmat-1m-recolor", "op": "recolor", "graph": "rmat", "n": 1 << 20, "ef": 16},
        # the repository's batch: mixed graphs of 100 to 200,000 vertices in one call
        {"name": "batch-256-mixed", "op": "batch", "graphs": 256, "n_min": 100, "n_max": 200000, "sizes": 3},
        # thousands of small graphs in one call
        {"name": "batch-4096-small", "op": "batch", "graphs": 4096, "n_min": 100, "n_max": 4000, "sizes": 5},
        # continuous-batching server: a burst of requests from pinned host buffers, every result polled
        {"name": "serve-24", "op": "serve", "graphs": 24, "n_min": 1000, "n_max": 200000, "sizes": 4},
    ]


def _log_uniform(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    op = rng.choice(["color"] * 6 + ["ordered"] * 2 + ["recolor", "levels", "batch", "batch", "serve"])
    if op == "batch":
        n_max = _log_uniform(rng, 400, 100000)
        return {"op": "batch", "graphs": _log_uniform(rng, 16, min(4096, max(17, 6000000 // n_max))), "n_min": 100,
                "n_max": n_max, "sizes": rng.randrange(1 << 20)}
    if op == "serve":
        return {"op": "serve", "graphs": rng.randrange(4, 25), "n_min": 1000, "n_max": _log_uniform(rng, 2000, 200000),
                "sizes": rng.randrange(1 << 20)}
    case = {"op": "color" if op in ("color", "ordered") else op}
    # (the levels of a mesh depend on nothing random)
    case["graph"] = rng.choice(["er", "rmat", "rmat"] + ([] if op == "levels" else ["stencil", "grid"]))
    top = 2000000 if op == "color" else 400000
    n = _log_uniform(rng, 300, top)
    if case["graph"] == "er":
        case["n"], case["degree"] = n, round(rng.uniform(4.0, 64.0 if n < 1000000 else 32.0), 2)
    elif case["graph"] == "rmat":
        case["n"], case["ef"] = n, rng.randrange(4, 17)
    elif case["graph"] == "stencil":
        side = n ** (1.0 / 3.0)
        case["nx"] = max(2, int(side * rng.uniform(0.5, 2.0)))
        case["ny"] = max(2, int(side * rng.uniform(0.5, 2.0)))
        case["nz"] = max(2, n // (case["nx"] * case["ny"]))
    else:
        case["nx"] = max(2, int(n ** 0.5 * rng.uniform(0.5, 2.0)))
        case["ny"] = max(2, n // case["nx"])
    if op == "ordered":
        case["mode"] = "ordered"
    if op in ("color", "ordered"):
        # (smallest last orders graphs with hubs; on a mesh it depends on nothing random)
        last = [gc.PRIORITY_SMALLEST_LAST] if case["graph"] in ("er", "rmat") else []
        case["priority"] = rng.choice([gc.PRIORITY_HASH] * 3 + [gc.PRIORITY_LARGEST_FIRST] + last)
    if op == "color" and rng.random() < 0.2:
        case["home"] = "host"
    return case


# ----------------------------------------------------------------------------------------------
# graphs

def _generator(seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(seed & ((1 << 62) - 1))
    return g


def _rmat_ids(levels, count, g):
    """`count` R-MAT id pairs of up to max(levels) bits: pair i gets levels[i] bits (or `levels` bits)."""
    u = torch.zeros(count, dtype=torch.int64, device=DEV)
    v = torch.zeros(count, dtype=torch.int64, device=DEV)
    most = int(levels) if isinstance(levels, int) else int(levels.max()) if count else 0
    for b in range(most):
        r = torch.rand(count, device=DEV, generator=g)
        ub = (r >= 0.76).to(torch.int64)
        vb = (((r >= 0.57) & (r < 0.76)) | (r >= 0.95)).to(torch.int64)
        if not isinstance(levels, int):
            take = (b < levels).to(torch.int64)
            ub *= take
            vb *= take
        u |= ub << b
        v |= vb << b
    return u, v


def _csr(n, u, v):
    """Symmetric, sorted, duplicate-free CSR (int32) of the pairs u != v."""
    keep = u != v
    u, v = u[keep], v[keep]
    key = torch.cat([u * n + v, v * n + u])
    del u, v, keep
    key = torch.unique(key)
    rowptr = torch.searchsorted(key, torch.arange(n + 1, device=DEV) * n).to(torch.int32)
    return rowptr, (key % n).to(torch.int32)


def _mesh(dims, corners):
    """Neighbours at distance 1 in every axis (corners: 27-point) or along one axis (5-point)."""
    n = math.prod(dims)
    ids = torch.arange(n, dtype=torch.int32, device=DEV)
    at, step, steps = [], 1, []
    for d in dims:
        at.append((ids // step) % d)
        steps.append(step)
        step *= d
    offs = [()]
    for _ in dims:
        offs = [o + (s,) for o in offs for s in (-1, 0, 1)]
    offs = [o for o in offs if any(o) and (corners or sum(abs(s) for s in o) == 1)]
    offs.sort(key=lambda o: sum(s * t for s, t in zip(o, steps)))
    nbr = torch.empty((n, len(offs)), dtype=torch.int32, device=DEV)
    ok = torch.ones((n, len(offs)), dtype=torch.bool, device=DEV)
    for k, o in enumerate(offs):
        nbr[:, k] = ids + sum(s * t for s, t in zip(o, steps))
        for s, a, d in zip(o, at, dims):
            if s:
                ok[:, k] &= (a + s >= 0) & (a + s < d)
    rowptr = torch.zeros(n + 1, dtype=torch.int32, device=DEV)
    rowptr[1:] = torch.cumsum(ok.sum(1), 0).to(torch.int32)
    return rowptr, torch.masked_select(nbr, ok)


def _graph(case, seed):
    g = _generator(seed)
    if case["graph"] == "stencil":
        return _mesh((case["nx"], case["ny"], case["nz"]), True)
    if case["graph"] == "grid":
        return _mesh((case["nx"], case["ny"]), False)
    n = case["n"]
    if case["graph"] == "er":
        m = int(n * case["degree"] / 2)
        u = torch.randint(n, (m,), device=DEV, generator=g)
        v = torch.randint(n, (m,), device=DEV, generator=g)
        return _csr(n, u, v)
    u, v = _rmat_ids(max(1, (n - 1).bit_length()), n * case["ef"], g)
    keep = (u < n) & (v < n)
    perm = torch.randperm(n, device=DEV, generator=g)
    u, v = perm[u[keep]], perm[v[keep]]
    return _csr(n, u, v)


def _sizes(case):
    """The graphs of a batch or a request stream: kind, vertices and edge attempts of each, from the case
    alone (even graphs ER of average degree 4..64, odd ones R-MAT of edge factor 8..16)."""
    r = random.Random(case["sizes"])
    got = []
    for k in range(case["graphs"]):
        n = _log_uniform(r, case["n_min"], case["n_max"])
        if k % 2 == 0:
            got.append(("er", n, int(n * r.uniform(4.0, 64.0) / 2)))
        else:
            got.append(("rmat", n, n * r.randint(8, 16)))
    return got


def _pack(case, seed):
    """The graphs of _sizes(case) in the packed layout of color_batch."""
    g = _generator(seed)
    sizes = _sizes(case)
    n = torch.tensor([s[1] for s in sizes], device=DEV)
    m = torch.tensor([s[2] for s in sizes], device=DEV)
    rm = torch.tensor([s[0] == "rmat" for s in sizes], device=DEV)
    lev = torch.tensor([max(1, (s[1] - 1).bit_length()) for s in sizes], device=DEV)
    vtx = torch.zeros(len(sizes) + 1, dtype=torch.int64, device=DEV)
    vtx[1:] = torch.cumsum(n, 0)
    total = int(vtx[-1])
    gid = torch.repeat_interleave(torch.arange(len(sizes), device=DEV), m)
    ng, isr = n[gid], rm[gid]
    u = (torch.rand(gid.numel(), device=DEV, generator=g, dtype=torch.float64) * ng).to(torch.int64)
    v = (torch.rand(gid.numel(), device=DEV, generator=g, dtype=torch.float64) * ng).to(torch.int64)
    at = torch.nonzero(isr).squeeze(1)
    ur, vr = _rmat_ids(lev[gid[at]], at.numel(), g)
    # ids permuted within each graph: vertices ordered by (graph, random)
    owner = torch.repeat_interleave(torch.arange(len(sizes), device=DEV), n)
    order = torch.argsort(owner.to(torch.float64) + torch.rand(total, device=DEV, generator=g, dtype=torch.float64) * 0.999)
    local = order - vtx[owner]
    base = vtx[gid[at]]
    fit = (ur < ng[at]) & (vr < ng[at])
    ur, vr = torch.where(fit, ur, 0), torch.where(fit, vr, 0)  # (0, 0) is dropped as a self-loop
    u[at], v[at] = local[base + ur], local[base + vr]
    keep = u != v
    u, v, gid = u[keep], v[keep], gid[keep]
    row = vtx[gid]
    key = torch.unique(torch.cat([((row + u) << 20) | v, ((row + v) << 20) | u]))
    first = torch.searchsorted(key, torch.arange(total + 1, device=DEV) << 20)
    edge = first[vtx]
    owner1 = torch.repeat_interleave(torch.arange(len(sizes), device=DEV), n + 1)
    pos = torch.arange(total + len(sizes), device=DEV)
    rowptr = (first[pos - owner1] - edge[owner1]).to(torch.int32)
    return vtx, edge, rowptr, (key & ((1 << 20) - 1)).to(torch.int32)


# ----------------------------------------------------------------------------------------------
# the passes

def prepare(case, seed):
    state = {"case": case, "seed": (seed * 0x9E3779B97F4A7C15 + 7) & ((1 << 63) - 1)}
    op = case["op"]
    if op == "batch":
        state["batch"] = _pack(case, seed)
    elif op == "serve":
        vtx, edge, rowptr, colidx = (a.cpu() for a in _pack(case, seed))
        graphs = []
        for k in range(case["graphs"]):
            a, b = int(vtx[k]) + k, int(vtx[k + 1]) + k + 1
            graphs.append((rowptr[a:b].clone().pin_memory().numpy(),
                           colidx[int(edge[k]):int(edge[k + 1])].clone().pin_memory().numpy()))
        state["requests"] = graphs
        state["server"] = gc.Server(pool_vertices=int(vtx[-1]) + 1024, pool_entries=int(edge[-1]) + 1024, mode="det")
    else:
        rowptr, colidx = _graph(case, seed)
        if case.get("home") == "host":
            rowptr, colidx = rowptr.cpu().pin_memory(), colidx.cpu().pin_memory()
            state["out"] = torch.empty(rowptr.numel() - 1, dtype=torch.int32).pin_memory()
        state["graph"] = (rowptr, colidx)
        if op == "recolor":
            state["colors"] = gc.color(rowptr, colidx, "det", state["seed"]).colors
    return state


def run(state):
    case, seed = state["case"], state["seed"]
    op = case["op"]
    if op == "batch":
        colors, ncolors, rounds = gc.color_batch(*state["batch"], mode="det", seed=seed)
        return [colors, ncolors, rounds]
    if op == "serve":
        server = state["server"]
        ids = [server.submit(rowptr, colidx, mode="det", seed=seed + k)
               for k, (rowptr, colidx) in enumerate(state["requests"])]
        done = [server.poll(i) for i in ids]
        return [d[0] for d in done] + [np.array([d[1] for d in done]), np.array([d[2] for d in done])]
    rowptr, colidx = state["graph"]
    if op == "levels":
        level, count, degeneracy = gc.smallest_last(rowptr, colidx)
        return [level, count, degeneracy]
    if op == "recolor":
        r = gc.recolor(rowptr, colidx, state["colors"], seed)
    else:
        r = gc.color(rowptr, colidx, case.get("mode", "det"), seed, out=state.get("out"),
                     options=gc.Options(priority=case.get("priority", gc.PRIORITY_HASH)))
    return [r.colors, r.ncolors, r.rounds]


def work(case):
    """Bytes of one pass: the CSR read once, the result written once.  The entries of random graphs are
    expected values (R-MAT loses about a tenth of its pairs to duplicates and self-loops, and the pairs
    past n when n is not a power of two)."""
    if case["op"] in ("batch", "serve"):
        n = entries = 0
        for kind, k, m in _sizes(case):
            n += k
            entries += min(k * (k - 1), int(2 * m * (1.0 if kind == "er" else 0.7)))
    elif case["graph"] == "er":
        n = case["n"]
        entries = int(n * case["degree"])
    elif case["graph"] == "rmat":
        n = case["n"]
        entries = int(2 * n * case["ef"] * (0.9 if n & (n - 1) == 0 else 0.75))
    elif case["graph"] == "stencil":
        n = case["nx"] * case["ny"] * case["nz"]
        entries = math.prod(3 * case[d] - 2 for d in ("nx", "ny", "nz")) - n
    else:
        n = case["nx"] * case["ny"]
        entries = 4 * n - 2 * (case["nx"] + case["ny"])
    extra = 4 * n if case["op"] == "recolor" else 0
    return {"bytes": 4 * (n + 1) + 4 * entries + 4 * n + extra, "flops": 0}


def exact(case, seed):
    """Every output is a whole number (colors, counts, rounds, levels): compared value by value."""
    return None
