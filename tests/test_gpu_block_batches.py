"""Which graphs of a batch a block each solves: batches of few graphs go to the
union where a block would take longer, large ones to the blocks, and both give
every graph's Kruskal forest."""
import numpy as np
import pytest
import torch

import oracle
from paper_2302_12199_gb300.mst import Solver

pytestmark = pytest.mark.gpu


def gnm(n, m, wmax, seed):
    rng = np.random.default_rng(seed)
    return n, *(rng.integers(0, n, m).astype(np.uint32) for _ in range(2)), \
        rng.integers(1, wmax, m, endpoint=True).astype(np.uint32)


def check(s, graphs, copies):
    """The graphs, `copies` times over in one batch, against Kruskal; the milliseconds and launches of block solves."""
    batch = graphs * copies
    off = np.cumsum([0] + [g[1].size for g in batch]).astype(np.uint64)
    t = [torch.from_numpy(np.concatenate([g[k] for g in batch]).view(np.int32)).to("cuda:0") for k in (1, 2, 3)]
    s.profile(True)
    ids, moff, tot = s.solve_batched(np.array([g[0] for g in batch], np.uint32), off, *t)
    launches = s.profile_stats()["base"][0]
    s.profile(False)
    ids, moff, tot = ids.cpu().numpy().view(np.uint32), moff.cpu().numpy(), tot.cpu().numpy().view(np.uint64)
    for i, g in enumerate(graphs):
        kid, ktot = oracle.kruskal(*g)
        for j in range(i, len(batch), len(graphs)):
            assert np.array_equal(ids[moff[j]:moff[j + 1]], kid) and int(tot[j]) == ktot, j
    return launches


# (vertices, edges, copies, a block each): a block's time against the union's, on either side, for each kind of block
@pytest.mark.parametrize("wmax", [255, 0xFFFFFFFF])
@pytest.mark.parametrize("n,m,copies,block", [(500, 4000, 1, True), (2048, 8192, 1, True), (8192, 40000, 1, False),
                                              (12288, 131072, 4, False), (65536, 131072, 1, False),
                                              (65536, 131072, 16, False), (28000, 65536, 16, False),
                                              (8192, 32768, 400, True), (20000, 60000, 300, True),
                                              (40000, 100000, 200, True)])
def test_small_batches_of_large_graphs(n, m, copies, block, wmax):
    for variant in ("boruvka", "filter"):
        s = Solver(0, variant=variant)
        try:
            assert (check(s, [gnm(n, m, wmax, n + m)], copies) > 0) == block
        finally:
            s.close()


def test_mixed_batches():
    """Graphs for blocks beside one for the union, when the blocks hold most edges and save more than they take, when
    they hold few, and when the longest would take longer than it saves."""
    small = [gnm(1500 + 20 * (i % 30), 6000, 255, i) for i in range(120)]
    large = [gnm(200000, 300000, 255, 99)]
    long = [gnm(12000, 60000, 255, 5), gnm(70000, 50000, 255, 6)]
    for graphs, block in ((small + large, True), (small[:20] + large, False), (long, False)):
        s = Solver(0)
        try:
            assert (check(s, graphs, 1) > 0) == block
        finally:
            s.close()


# as the batch of one graph of each size in test_gpu_block.py, often enough over that the blocks take them
@pytest.mark.parametrize("wmax", [255, 70000, 0xFFFFFFFF])
def test_blocks_at_their_edges_in_a_large_batch(wmax):
    sizes = [(1, 3), (2, 1), (300, 1023), (600, 1025), (700, 2049), (6146, 30000), (6147, 30001), (12288, 60001),
             (12289, 60002), (28416, 90000), (28417, 90001), (28672, 100000), (28673, 100003), (57344, 130001),
             (57345, 130002), (65535, 90001), (65536, 131000), (5, 0), (40, 4099)]
    graphs = [gnm(n, m, wmax, 31 * i + 7) for i, (n, m) in enumerate(sizes)]
    s = Solver(0)
    try:
        assert check(s, graphs, 30) > 0
    finally:
        s.close()
