"""Timed cases of the minimum-spanning-forest solver, through its public entry points.

Each case is one call a program makes: mst_solve on a graph in device memory
(Solver.solve), mst_solve_batched on many graphs (Solver.solve_batched) or
mst_solve_host_many on graphs in page-locked host memory
(Solver.solve_host_many_ptr).  The graph families are those of the benchmark
(GNM, 2D and 3D random geometric, 2D grid, RMAT, mixed batches), drawn on the
GPU with torch from the case's seed.  A program keeps one solver handle and
gives it one graph after another, so the states of a case share a handle.
"""
from __future__ import annotations

import json
import math
import weakref

import torch

from paper_2302_12199_gb300.mst import Forest, Solver

DEV = torch.device("cuda", 0)

# ------------------------------------------------------------------- cases

_LISTED = [
    # the smallest call: one graph of the served mix's lower end, alone (launches and readbacks only)
    dict(name="gnm_small", kind="gnm", n=256, m=2048, variant="boruvka", wmax=255),
    # GNM of the benchmark: input in L2, plain Borůvka, many ties
    dict(name="gnm", kind="gnm", n=1 << 16, m=1 << 20, variant="boruvka", wmax=255),
    # a dense mid-size graph of odd sizes, the variant left to the solver, weights over the whole 32 bits
    dict(name="gnm_auto_odd", kind="gnm", n=250007, m=4000037, variant="auto", wmax=0xFFFFFFFF),
    # geometric graphs of the benchmark: ids in Morton order of the grid cells, 32-bit weights
    dict(name="rgg2d", kind="rgg2d", n=1 << 22, deg=8.0, variant="boruvka", wmax=0xFFFFFFFF),
    dict(name="rgg3d", kind="rgg3d", n=1 << 21, deg=8.0, variant="boruvka", wmax=0xFFFFFFFF),
    # 4-neighbour grid of the benchmark, row-major ids
    dict(name="grid2d", kind="grid2d", rows=2048, cols=2048, variant="boruvka", wmax=255),
    # the headline: RMAT scale 24, 2^28 edges, Filter-Borůvka
    dict(name="rmat_filter", kind="rmat", n=1 << 24, m=1 << 28, variant="filter", wmax=255),
    # a smaller RMAT of odd sizes under Filter-Borůvka
    dict(name="rmat_filter_odd", kind="rmat", n=1500007, m=20000003, variant="filter", wmax=255),
    # plain Borůvka on a heavy-tailed graph
    dict(name="rmat_boruvka", kind="rmat", n=1 << 22, m=1 << 26, variant="boruvka", wmax=255),
    # the batched benchmark: 4096 uneven graphs in one call, size tables on the device, the tuned quantile
    dict(name="batch", kind="batch", graphs=4096, log_hi=16, variant="filter", quantile=0.25, tables="device"),
    # one batch of the served stream: few graphs up to 2^20 vertices, the server's configuration and host tables
    dict(name="batch_served", kind="batch", graphs=48, log_hi=20, variant="filter", quantile=0.125, tables="host"),
    # graphs in page-locked host memory, solved in sequence (copies overlap solves)
    dict(name="host_many", kind="host", n=1 << 20, m=1 << 23, graphs=3, variant="filter", wmax=255),
]


def listed():
    return [dict(c) for c in _LISTED]


def _log_uniform(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more case of the same families, options and size ranges."""
    kind = rng.choice(["gnm", "gnm", "rgg2d", "rgg3d", "grid2d", "rmat", "rmat", "rmat", "batch", "batch", "host"])
    wmax = rng.choice([255, 0xFFFFFFFF])
    if kind == "gnm":
        n = _log_uniform(rng, 1 << 8, 1 << 20)
        m = max(1, int(n * rng.uniform(4.0, 32.0) / 2))
        return dict(kind="gnm", n=n, m=m, variant=rng.choice(["boruvka", "auto"]), wmax=wmax)
    if kind in ("rgg2d", "rgg3d"):
        return dict(kind=kind, n=_log_uniform(rng, 1 << 10, 1 << (22 if kind == "rgg2d" else 21)), deg=8.0,
                    variant="boruvka", wmax=wmax)
    if kind == "grid2d":
        return dict(kind="grid2d", rows=_log_uniform(rng, 16, 2048), cols=_log_uniform(rng, 16, 2048),
                    variant="boruvka", wmax=255)
    if kind == "rmat":
        variant = rng.choice(["filter", "filter", "boruvka"])
        n = _log_uniform(rng, 1 << 12, 1 << (24 if variant == "filter" else 22))
        return dict(kind="rmat", n=n, m=int(n * rng.uniform(8.0, 16.0)), variant=variant, wmax=255)
    if kind == "host":
        n = _log_uniform(rng, 1 << 12, 1 << 21)
        return dict(kind="host", n=n, m=int(n * rng.uniform(4.0, 16.0)), graphs=rng.randint(2, 4), variant="filter",
                    wmax=255)
    if rng.random() < 0.5:
        return dict(kind="batch", graphs=_log_uniform(rng, 64, 4096), log_hi=16, variant="filter",
                    quantile=rng.choice([0.25, 0.125]), tables="device")
    return dict(kind="batch", graphs=_log_uniform(rng, 2, 64), log_hi=20,
                variant=rng.choice(["filter", "filter", "boruvka"]), quantile=0.125, tables="host")


# -------------------------------------------------------------- generators


def _gen(seed, salt=0):
    g = torch.Generator(device=DEV)
    g.manual_seed((int(seed) * 1000003 + salt * 7919 + 17) & 0x7FFFFFFFFFFFFFFF)
    return g


def _weights(gen, m, wmax):
    """Uniform in [1, wmax], as the int32 tensor that holds the uint32 bits."""
    if wmax < (1 << 31):
        return torch.randint(1, wmax + 1, (m,), generator=gen, device=DEV, dtype=torch.int32)
    x = torch.randint(1, wmax + 1, (m,), generator=gen, device=DEV, dtype=torch.int64)
    return torch.where(x >= (1 << 31), x - (1 << 32), x).to(torch.int32)


def _gnm(gen, n, m):
    """m uniform endpoint pairs without self-loops, duplicates kept."""
    u = torch.randint(0, n, (m,), generator=gen, device=DEV, dtype=torch.int32)
    v = torch.randint(0, max(1, n - 1), (m,), generator=gen, device=DEV, dtype=torch.int32)
    return u, v + (v >= u).to(torch.int32)


def _rmat_ends(gen, levels, m):
    """Ends of m RMAT edges with quadrant probabilities 0.57, 0.19, 0.19, 0.05; levels: a number, or per edge."""
    deep = levels if isinstance(levels, int) else int(levels.max())
    u = torch.zeros(m, dtype=torch.int32, device=DEV)
    v = torch.zeros(m, dtype=torch.int32, device=DEV)
    for lo in range(0, m, 1 << 26):  # bounded temporaries
        hi = min(m, lo + (1 << 26))
        a, b = u[lo:hi], v[lo:hi]
        for k in range(deep):
            r = torch.rand(hi - lo, generator=gen, device=DEV)
            ub, vb = r >= 0.76, ((r >= 0.57) & (r < 0.76)) | (r >= 0.95)
            if not isinstance(levels, int):  # an edge of a smaller graph stops earlier
                on = levels[lo:hi] > k
                a.copy_(torch.where(on, 2 * a + ub, a))
                b.copy_(torch.where(on, 2 * b + vb, b))
            else:
                a.mul_(2).add_(ub)
                b.mul_(2).add_(vb)
    return u, v


def _rmat(gen, n, m):
    """RMAT with randomly permuted ids (folded into 0..n-1); self-loops and duplicates kept."""
    u, v = _rmat_ends(gen, max(1, math.ceil(math.log2(n))), m)
    perm = torch.randperm(n, generator=gen, device=DEV).to(torch.int32)
    for x in (u, v):
        for lo in range(0, m, 1 << 26):
            part = x[lo:lo + (1 << 26)]
            part.copy_(perm[part.remainder(n).long()])
    return u, v


def _morton(xs):
    """Interleaved bits of the integer coordinates (int64 tensors)."""
    code = torch.zeros_like(xs[0])
    bits = max(1, int(max(int(x.max()) for x in xs)).bit_length())
    for b in range(bits):
        for d, x in enumerate(xs):
            code |= ((x >> b) & 1) << (b * len(xs) + d)
    return code


def _rgg(gen, dim, ns, deg):
    """Random geometric graphs of ns[i] uniform points (expected degree deg), ids by grid cell in Morton order.

    Returns (u, v, graph) with graph-local ids, edges grouped by graph and, in it, by their first end."""
    ns = [int(x) for x in ns]
    r = [math.sqrt(deg / (math.pi * n)) if dim == 2 else (3.0 * deg / (4.0 * math.pi * n)) ** (1.0 / 3.0) for n in ns]
    cells = [max(1, int(1.0 / min(1.0, x))) for x in r]
    side = [1 << max(0, (c - 1).bit_length()) for c in cells]
    nt = torch.tensor(ns, device=DEV)
    first = torch.cumsum(nt, 0) - nt
    graph = torch.repeat_interleave(torch.arange(len(ns), device=DEV), nt)
    pt = torch.rand(graph.numel(), dim, generator=gen, device=DEV)
    gc = torch.tensor(cells, device=DEV)[graph]
    space = torch.tensor([s ** dim for s in side], device=DEV)
    base = torch.cumsum(space, 0) - space
    cell = [torch.minimum((pt[:, d] * gc).long(), gc - 1) for d in range(dim)]
    key, order = torch.sort(base[graph] + _morton(cell), stable=True)
    pt, cell = pt[order], [c[order] for c in cell]  # (points of a graph stay in its range)
    start = torch.zeros(int(space.sum()) + 1, dtype=torch.int64, device=DEV)
    start[1:] = torch.cumsum(torch.bincount(key, minlength=int(space.sum())), 0)
    r2 = torch.tensor([x * x for x in r], device=DEV)[graph]
    me = torch.arange(key.numel(), device=DEV)
    ends = []
    offsets = [()]
    for _ in range(dim):
        offsets = [o + (d,) for o in offsets for d in (-1, 0, 1)]
    for off in (o for o in offsets if o >= (0,) * dim):  # each pair of cells once
        nb = [c + o for c, o in zip(cell, off)]
        ok = torch.ones_like(me, dtype=torch.bool)
        for x in nb:
            ok &= (x >= 0) & (x < gc)
        code = base[graph] + _morton([x.clamp(min=0) for x in nb])
        code = torch.where(ok, code, 0)
        lo = me + 1 if not any(off) else start[code]
        cnt = torch.where(ok, start[code + 1] - lo, 0)
        i = torch.repeat_interleave(me, cnt)
        j = torch.arange(i.numel(), device=DEV) - torch.repeat_interleave(torch.cumsum(cnt, 0) - cnt, cnt) + lo[i]
        near = ((pt[i] - pt[j]) ** 2).sum(1) < r2[i]
        ends.append((i[near], j[near]))
    i, j = torch.cat([e[0] for e in ends]), torch.cat([e[1] for e in ends])
    i, order = torch.sort(i, stable=True)
    g = graph[i]
    return (i - first[g]).to(torch.int32), (j[order] - first[g]).to(torch.int32), g


def _grid2d(rows, cols):
    """Edges of the 4-neighbour grid: each vertex's right and down edge, row by row."""
    v = torch.arange(rows * cols, dtype=torch.int32, device=DEV)
    right, down = v % cols < cols - 1, v < (rows - 1) * cols
    u = torch.stack([v, v], 1).reshape(-1)
    to = torch.stack([v + 1, v + cols], 1).reshape(-1)
    keep = torch.stack([right, down], 1).reshape(-1)
    return u[keep], to[keep]


def _graph(case, seed):
    """(n, src, dst, w) of a single-graph case, on the GPU."""
    gen = _gen(seed)
    kind = case["kind"]
    if kind == "rmat" or kind == "host":
        n, (u, v) = case["n"], _rmat(gen, case["n"], case["m"])
    elif kind == "gnm":
        n, (u, v) = case["n"], _gnm(gen, case["n"], case["m"])
    elif kind == "grid2d":
        n, (u, v) = case["rows"] * case["cols"], _grid2d(case["rows"], case["cols"])
    else:
        n = case["n"]
        u, v, _ = _rgg(gen, 2 if kind == "rgg2d" else 3, [n], case["deg"])
    return n, u.contiguous(), v.contiguous(), _weights(gen, u.numel(), case["wmax"])


def _batch(case, seed):
    """(n per graph, edge offsets, src, dst, w): graph g is GNM (average degree 4 to 32), 2D geometric (degree 8) or
    RMAT (degree 16) for g mod 3 = 0, 1, 2; n log-uniform in [2^8, 2^log_hi], one size from each of as many strata as
    there are graphs and in random order, so that every batch of a case has as many vertices."""
    gen, count = _gen(seed), case["graphs"]
    strata = (torch.arange(count, device=DEV, dtype=torch.float64) + 0.5) / count
    strata = strata[torch.randperm(count, generator=gen, device=DEV)]
    n = (2.0 ** (8 + (case["log_hi"] - 8) * strata)).long()
    g = torch.arange(count, device=DEV)
    m = torch.zeros(count, dtype=torch.int64, device=DEV)
    deg = 4 + 28 * torch.rand(count, generator=gen, device=DEV)
    m = torch.where(g % 3 == 0, (n * deg / 2).long(), torch.where(g % 3 == 2, 8 * n, m))
    ru = None
    if count > 1:
        ru, rv, rg = _rgg(gen, 2, n[1::3].tolist(), 8.0)
        m[1::3] = torch.bincount(rg, minlength=n[1::3].numel())
    off = torch.zeros(count + 1, dtype=torch.int64, device=DEV)
    off[1:] = torch.cumsum(m, 0)
    total = int(off[-1])
    src = torch.empty(total, dtype=torch.int32, device=DEV)
    dst = torch.empty(total, dtype=torch.int32, device=DEV)
    for kind in range(3):
        ids = g[kind::3]
        if ids.numel() == 0:
            continue
        of = torch.repeat_interleave(ids, m[ids])  # graph of each of this family's edges
        at = off[of] + torch.arange(of.numel(), device=DEV) - torch.repeat_interleave(
            torch.cumsum(m[ids], 0) - m[ids], m[ids])
        nn = n[of]
        if kind == 0:
            u = (torch.rand(of.numel(), generator=gen, device=DEV, dtype=torch.float64) * nn).long()
            v = (torch.rand(of.numel(), generator=gen, device=DEV, dtype=torch.float64) * (nn - 1)).long()
            v += v >= u
        elif kind == 1:
            u, v = ru, rv
        else:
            levels = torch.ceil(torch.log2(n.double())).to(torch.int32)
            u, v = _rmat_ends(gen, levels[of], of.numel())
            # ids permuted within each graph: ranks of random keys, graph by graph
            rank = torch.zeros(int(n.sum()), dtype=torch.int64, device=DEV)
            first = torch.cumsum(n, 0) - n
            own = torch.repeat_interleave(g, n)
            order = torch.argsort(own.double() + torch.rand(own.numel(), generator=gen, device=DEV,
                                                            dtype=torch.float64))
            rank[order] = torch.arange(own.numel(), device=DEV) - first[own]
            u, v = rank[first[of] + u % nn], rank[first[of] + v % nn]
        src[at], dst[at] = u.to(torch.int32), v.to(torch.int32)
    return n, off, src, dst, _weights(gen, total, 255)


# ------------------------------------------------------- what a program has

_SOLVERS = weakref.WeakValueDictionary()  # one handle per case, as long as a state of the case lives


def _solver(case):
    key = json.dumps({k: v for k, v in case.items() if k != "name"}, sort_keys=True)
    s = _SOLVERS.get(key)
    if s is None:
        s = Solver(0, variant=case["variant"], **({"pivot_quantile": case["quantile"]} if "quantile" in case else {}))
        _SOLVERS[key] = s
    return s


def _capacity(n, m):
    return max(1, min(m, max(n - 1, 0)))


def prepare(case, seed):
    state = {"kind": case["kind"], "solver": _solver(case)}
    if case["kind"] == "batch":
        n, off, src, dst, w = _batch(case, seed)
        state.update(src=src, dst=dst, w=w, capacity=int(n.sum()))
        # where the program keeps the forests (a call's ids live until the next call only in a server's slot)
        state["forests"] = torch.zeros(state["capacity"], dtype=torch.int32, device=DEV)
        if case["tables"] == "device":
            state.update(n=n.to(torch.int32), off=off)
        else:
            import numpy as np
            state.update(n=n.cpu().numpy().astype(np.uint32), off=off.cpu().numpy().astype(np.uint64))
    elif case["kind"] == "host":
        state["graphs"], state["keep"] = [], []
        for k in range(case["graphs"]):
            n, *edges = _graph(case, seed * 16 + k)
            pinned = [torch.empty(e.numel(), dtype=torch.int32, pin_memory=True).copy_(e) for e in edges]
            ids = torch.empty(_capacity(n, edges[0].numel()), dtype=torch.int32, pin_memory=True).zero_()
            state["graphs"].append((n, edges[0].numel(), *(p.data_ptr() for p in pinned), ids.data_ptr()))
            state["keep"].append((pinned, ids))
    else:
        n, src, dst, w = _graph(case, seed)
        ids = torch.zeros(_capacity(n, src.numel()), dtype=torch.int32, device=DEV)
        out = Forest(ids, torch.zeros(1, dtype=torch.int32, device=DEV), torch.zeros(1, dtype=torch.int64, device=DEV))
        state.update(n=n, src=src, dst=dst, w=w, out=out)
    torch.cuda.synchronize()
    return state


def run(state):
    solver = state["solver"]
    if state["kind"] == "batch":
        ids, off, totals = solver.solve_batched(state["n"], state["off"], state["src"], state["dst"], state["w"],
                                                capacity=state["capacity"])
        k = int(off[-1])
        state["forests"][:k].copy_(ids[:k])
        return {"ids": state["forests"], "off": off, "totals": totals}
    if state["kind"] == "host":
        res = solver.solve_host_many_ptr(state["graphs"])
        return {"ids": [k[1] for k in state["keep"]], "count": [c for c, _ in res], "total": [t for _, t in res]}
    out = solver.solve(state["n"], state["src"], state["dst"], state["w"], out=state["out"])
    return {"ids": out.ids, "count": out.count, "total": out.total}


def _sizes(case):
    """(vertices, edges) of a case; expected numbers where the seed decides."""
    kind = case["kind"]
    if kind == "batch":
        n = case["graphs"] * (2.0 ** case["log_hi"] - 2.0 ** 8) / ((case["log_hi"] - 8) * math.log(2.0))
        return n, 7.0 * n  # average degrees 18, 8 and 16 in equal parts
    if kind == "grid2d":
        return case["rows"] * case["cols"], 2 * case["rows"] * case["cols"] - case["rows"] - case["cols"]
    if kind in ("rgg2d", "rgg3d"):
        return case["n"], case["n"] * case["deg"] / 2
    k = case.get("graphs", 1)
    return k * case["n"], k * case["m"]


def work(case):
    """Each edge (two ends and a weight, 12 bytes) read once, the forest's ids (4 bytes) written once."""
    n, m = _sizes(case)
    return {"bytes": 12.0 * m + 4.0 * min(n, m), "flops": 0.0}


# -------------------------------------------------------------------- exact


def _forest(n, u, v, w):
    """Ids of the minimum spanning forest under the order (w, id), and its weight: Borůvka rounds in 64-bit torch."""
    w = w.long() & 0xFFFFFFFF
    a, b = u.long(), v.long()
    ids = torch.nonzero(a != b).reshape(-1)
    a, b = a[ids], b[ids]
    key = (w[ids] << 29) | ids
    top = (1 << 62)
    me = torch.arange(n, device=DEV)
    chosen = []
    while key.numel():
        best = torch.full((n,), top, dtype=torch.int64, device=DEV)
        best.scatter_reduce_(0, a, key, "amin")
        best.scatter_reduce_(0, b, key, "amin")
        of_a, of_b = best[a] == key, best[b] == key
        chosen.append(key[of_a | of_b] & ((1 << 29) - 1))
        parent = me.clone()
        parent[a[of_a]] = b[of_a]
        parent[b[of_b]] = a[of_b]
        parent = torch.where((parent[parent] == me) & (me < parent), me, parent)  # 2-cycles
        while True:
            up = parent[parent]
            if torch.equal(up, parent):
                break
            parent = up
        a, b = parent[a], parent[b]
        live = a != b
        a, b, key = a[live], b[live], key[live]
    got = torch.sort(torch.cat(chosen)).values if chosen else torch.zeros(0, dtype=torch.int64, device=DEV)
    return got, w[got].sum()


def exact(case, seed):
    """What run() returns for these inputs, by plain torch in 64 bits."""
    if case["kind"] == "batch":
        n, off, src, dst, w = _batch(case, seed)
        of = torch.repeat_interleave(torch.arange(n.numel(), device=DEV), off[1:] - off[:-1])
        first = (torch.cumsum(n, 0) - n)[of]
        got, _ = _forest(int(n.sum()), src + first, dst + first, w)
        totals = torch.zeros(n.numel(), dtype=torch.int64, device=DEV)
        totals.scatter_add_(0, of[got], w[got].long() & 0xFFFFFFFF)
        ids = torch.zeros(int(n.sum()), dtype=torch.int32, device=DEV)
        ids[:got.numel()] = (got - off[of[got]]).to(torch.int32)
        return {"ids": ids, "off": torch.searchsorted(got, off), "totals": totals}
    graphs = [_graph(case, seed * 16 + k) for k in range(case["graphs"])] if case["kind"] == "host" else [
        _graph(case, seed)]
    ids, counts, sums = [], [], []
    for n, u, v, w in graphs:
        got, total = _forest(n, u, v, w)
        out = torch.zeros(_capacity(n, u.numel()), dtype=torch.int32, device=DEV)
        out[:got.numel()] = got.to(torch.int32)
        ids.append(out)
        counts.append(got.numel())
        sums.append(int(total))
    if case["kind"] == "host":
        return {"ids": ids, "count": counts, "total": sums}
    return {"ids": ids[0], "count": torch.tensor(counts, dtype=torch.int32), "total": torch.tensor(sums)}
