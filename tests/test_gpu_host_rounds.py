"""Passes that the default configuration no longer reaches on small or plain
inputs: the one-launch rounds at sizes that a single block would solve, and the
tile shapes and the base case of rounds that the host drives.  Every test checks
that what it names was launched; every forest against Kruskal."""
import functools

import numpy as np
import pytest
import torch

import oracle
from paper_2302_12199_gb300 import workloads as W
from paper_2302_12199_gb300.mst import Solver

pytestmark = pytest.mark.gpu


def solve(s, g, shift=0):
    t = [torch.zeros(g.m + shift, dtype=torch.int32, device="cuda:0") for _ in range(3)]
    for x, a in zip(t, (g.src, g.dst, g.w)):
        x[shift:] = torch.from_numpy(a.view(np.int32)).to("cuda:0")
    return s.solve(g.n, *(x[shift:] for x in t)).to_host()


def launched(s):
    return {k for k, v in s.profile_stats().items() if v[0]}


def random_graph(n, m, wmax, seed):
    """Random edges (self-loops and duplicates among them) over half a random path, so that chains are long."""
    rng = np.random.default_rng(seed)
    src = rng.integers(0, n, m)
    dst = np.where(rng.random(m) < 0.5, np.minimum(src + 1, n - 1), rng.integers(0, n, m))
    w = np.where(rng.random(m) < 0.3, 1 + src % wmax, rng.integers(1, wmax + 1, m))
    return W.Graph(n, src.astype(np.uint32), dst.astype(np.uint32), w.astype(np.uint32))


# one edge; around a tile of 512 and of 2048 edges; around the one-block finish (4096 edges and vertices), from the start
# (a grid of one block) and after some rounds
@pytest.mark.parametrize("wmax", [255, 0xFFFFFFFF])
@pytest.mark.parametrize("n,m", [(2, 1), (512, 511), (513, 512), (600, 513), (2048, 2049), (4096, 4096), (4097, 4096),
                                 (4096, 4097), (12288, 32768)])
def test_small_graphs_in_one_launch_rounds(n, m, wmax):
    g = random_graph(n, m, wmax, 17 * n + m)
    kid, ktot = oracle.kruskal(g.n, g.src, g.dst, g.w)
    for cfg in (dict(), dict(variant="filter", filter_min_edges=256, pivot_sample=1024),
                dict(variant="filter", filter_min_edges=256, pivot_sample=1024, filter_plan=0)):
        s = Solver(0, base_case=0, **cfg)
        try:
            s.profile(True, classes=[])
            for shift in (0, 1):
                ids, tot = solve(s, g, shift)
                assert np.array_equal(ids, kid) and tot == ktot, (cfg, shift)
            assert "graph" in launched(s) and "base" not in launched(s)
        finally:
            s.close()


@functools.lru_cache(None)
def shape_case(name):
    g, cfg = {
        # lists long enough for the persistent bulk-copy relabel in every shape that has one; packed keys
        "rmat": lambda: (W.rmat(18, 3_000_000, 51), dict(variant="boruvka")),
        "rmat_filter": lambda: (W.rmat(17, 1_500_000, 54), dict(variant="filter", filter_min_edges=1 << 17)),
        # 32-bit weights: unpacked keys, the walking hook
        "rgg2d": lambda: (W.rgg(2, 1 << 16, 8.0, 52), dict(variant="boruvka")),
        # deepest pointer jumping, ragged tiles
        "path": lambda: (W.Graph(100_001, np.arange(100_000, dtype=np.uint32),
                                 np.arange(1, 100_001, dtype=np.uint32),
                                 (np.arange(100_000, dtype=np.uint32) % 13 + 1).astype(np.uint32)),
                         dict(variant="boruvka")),
    }[name]()
    return g, cfg, oracle.kruskal(g.n, g.src, g.dst, g.w)


@pytest.mark.parametrize("items", [4, 8, 16])
@pytest.mark.parametrize("threads", [128, 256, 512])
@pytest.mark.parametrize("options", [("block_threads", "items_per_thread"),
                                     ("relabel_block_threads", "relabel_items_per_thread")])
def test_every_shape_of_host_driven_rounds(options, threads, items):
    for name in ("rmat", "rmat_filter", "rgg2d", "path"):
        g, cfg, (kid, ktot) = shape_case(name)
        s = Solver(0, graph_rounds=0, base_case=0, **dict(zip(options, (threads, items))), **cfg)
        try:
            s.profile(True, classes=[])
            for shift in (0, 1):
                ids, tot = solve(s, g, shift)
                assert np.array_equal(ids, kid) and tot == ktot, (name, shift)
            assert launched(s) >= {"hook", "relabel_min", "jump"} and "graph" not in launched(s)
        finally:
            s.close()


@pytest.mark.parametrize("family", ["gnm", "rmat", "rgg2", "path", "star"])
def test_base_case_of_host_driven_rounds(family):
    """The single-block base case finishes the last rounds, or nothing does."""
    g = {
        "gnm": lambda: W.gnm(3000, 20000, 51),
        "rmat": lambda: W.rmat(13, 60000, 52),
        "rgg2": lambda: W.rgg(2, 20000, 8.0, 53),
        "path": lambda: W.Graph(5000, np.arange(4999, dtype=np.uint32), np.arange(1, 5000, dtype=np.uint32),
                                (np.arange(4999, dtype=np.uint32) % 7 + 1).astype(np.uint32)),
        "star": lambda: W.Graph(7000, np.zeros(6999, dtype=np.uint32), np.arange(1, 7000, dtype=np.uint32),
                                (np.arange(6999, dtype=np.uint32) % 7 + 1).astype(np.uint32)),
    }[family]()
    kid, ktot = oracle.kruskal(g.n, g.src, g.dst, g.w)
    for variant in ("boruvka", "filter"):
        for base in (0, 1):
            s = Solver(0, variant=variant, graph_rounds=0, base_case=base, filter_min_edges=1 << 10)
            try:
                s.profile(True, classes=[])
                ids, tot = solve(s, g)
                assert np.array_equal(ids, kid) and tot == ktot, (variant, base)
                assert "graph" not in launched(s)
                if base == 0:
                    assert "base" not in launched(s)
                elif family in ("rgg2", "path"):  # (denser graphs keep too many edges until their last round)
                    assert "base" in launched(s), variant
            finally:
                s.close()
