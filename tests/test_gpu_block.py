"""Graphs solved by one block each (in batches, and small graphs alone), at the
sizes where the blocks' shared memory, tiles and key widths end; every forest
against Kruskal."""
import numpy as np
import pytest
import torch

import oracle
from paper_2302_12199_gb300.mst import MstError, Solver

pytestmark = pytest.mark.gpu

KINDS = ["mixed", "path", "star", "equal", "apart"]


def graph(kind, n, m, wmax, seed):
    rng = np.random.default_rng(seed)
    if kind == "path":  # one long hooking chain under random heavier edges
        k = min(m, n - 1)
        src = np.concatenate([np.arange(k), rng.integers(0, n, m - k)])
        dst = np.concatenate([np.arange(1, k + 1), rng.integers(0, n, m - k)])
        w = np.concatenate([1 + np.arange(k) * (wmax // 2) // max(k, 1), wmax // 2 + rng.integers(0, wmax // 2, m - k)])
        p = rng.permutation(m)
        src, dst, w = src[p], dst[p], w[p]
    elif kind == "star":
        src, dst, w = np.zeros(m, np.int64), rng.integers(0, n, m), rng.integers(1, wmax + 1, m)
    elif kind == "apart":  # most vertices without edges, and components of their own
        src = rng.integers(0, max(1, n // 8), m) * 8 % n
        dst, w = np.minimum(src + 8 * rng.integers(0, 2, m), n - 1), rng.integers(1, wmax + 1, m)
    else:
        src, dst, w = rng.integers(0, n, m), rng.integers(0, n, m), rng.integers(1, wmax + 1, m)
        if kind == "equal":
            w[:] = wmax
    return n, src.astype(np.uint32), dst.astype(np.uint32), w.astype(np.uint32)


def solve_batch(s, graphs, shift=0):
    dev = torch.device("cuda", 0)
    n = np.array([g[0] for g in graphs], np.uint32)
    off = np.zeros(len(graphs) + 1, np.uint64)
    np.cumsum([g[1].size for g in graphs], out=off[1:])
    t = []
    for k in (1, 2, 3):
        a = np.concatenate([g[k] for g in graphs])
        x = torch.zeros(a.size + shift, dtype=torch.int32, device=dev)
        x[shift:] = torch.from_numpy(a.view(np.int32)).to(dev)
        t.append(x[shift:])
    ids, moff, tot = s.solve_batched(n, off, *t)
    return ids.cpu().numpy().view(np.uint32), moff.cpu().numpy(), tot.cpu().numpy().view(np.uint64)


def check(s, graphs, shift=0):
    ids, moff, tot = solve_batch(s, graphs, shift)
    for g, (n, src, dst, w) in enumerate(graphs):
        kid, ktot = oracle.kruskal(n, src, dst, w)
        assert np.array_equal(ids[moff[g]:moff[g + 1]], kid) and int(tot[g]) == ktot, g


@pytest.mark.parametrize("wmax", [255, 70000, 0xFFFFFFFF])
@pytest.mark.parametrize("kind", KINDS)
def test_batches_at_the_blocks_edges(kind, wmax):
    """Vertices around the small blocks' limit (12288), around what 32- and
    64-bit minima fill shared memory with (57344, 28672, 6146) and at the label
    limit (65536); edges around a tile and where the pivot starts; a graph too
    large for a block, an empty one and one without edges among them."""
    sizes = [(1, 3), (2, 1), (300, 1023), (600, 1025), (700, 2049), (6146, 30000), (6147, 30001), (12288, 60001),
             (12289, 60002), (28672, 100000), (28673, 100003), (57344, 130001), (57345, 130002), (65535, 90001),
             (65536, 131000), (5, 0), (65537, 70000), (40, 4099)]
    graphs = [graph(kind, n, m, wmax, 31 * i + 7) if m else (n, *(np.zeros(0, np.uint32),) * 3)
              for i, (n, m) in enumerate(sizes)]
    for cfg in (dict(), dict(variant="filter", filter_min_edges=1 << 10, pivot_sample=4096)):
        s = Solver(0, **cfg)
        try:
            for shift in (0, 3):
                check(s, graphs, shift)
        finally:
            s.close()


@pytest.mark.parametrize("wmax", [255, 0xFFFFFFFF])
@pytest.mark.parametrize("n,m", [(1, 5), (2, 1), (33, 32), (1024, 4095), (1025, 4097), (4096, 32768), (12288, 32767),
                                 (12289, 32768), (300, 32769)])
def test_small_graphs_alone(n, m, wmax):
    """One graph in one block, up to its limits and just past them."""
    dev = torch.device("cuda", 0)
    s = Solver(0)
    try:
        for kind in KINDS:
            _, src, dst, w = graph(kind, n, m, wmax, n + m)
            kid, ktot = oracle.kruskal(n, src, dst, w)
            t = [torch.from_numpy(a.view(np.int32)).to(dev) for a in (src, dst, w)]
            ids, tot = s.solve(n, *t).to_host()
            assert np.array_equal(ids, kid) and tot == ktot, kind
    finally:
        s.close()


def test_batch_vertex_out_of_range():
    """A vertex id past its graph's count, in a graph a block solves, fails the call; the handle then solves."""
    graphs = [graph("mixed", 500, 3000, 255, 1), graph("mixed", 20000, 90000, 255, 2)]
    s = Solver(0)
    try:
        for bad in (0, 1):
            n, src, dst, w = graphs[bad]
            broken = [g if i != bad else (n, src, np.where(np.arange(dst.size) == 77, n, dst).astype(np.uint32), w)
                      for i, g in enumerate(graphs)]
            with pytest.raises(MstError) as e:
                solve_batch(s, broken)
            assert e.value.status == 2
            check(s, graphs)
    finally:
        s.close()
