"""Rounds that end by the lightest edge between each two components, at the
sizes where that begins and ends; every forest against Kruskal."""
import numpy as np
import pytest
import torch

import oracle
from paper_2302_12199_gb300.mst import Solver

pytestmark = pytest.mark.gpu


def clusters(k, size, between, wmax, seed):
    """k stars of `size` vertices, which the first round contracts, and `between` random heavier edges (parallel ones
    and edges inside a star among them), shuffled."""
    rng = np.random.default_rng(seed)
    n = k * size
    leaf = np.arange(n)[np.arange(n) % size != 0]
    src = np.concatenate([leaf, rng.integers(0, n, between)])
    dst = np.concatenate([leaf - leaf % size, rng.integers(0, n, between)])
    w = np.concatenate([np.ones(leaf.size, np.int64), rng.integers(2, wmax + 1, between)])
    p = rng.permutation(src.size)
    return n, src[p].astype(np.uint32), dst[p].astype(np.uint32), w[p].astype(np.uint32)


# components after the first round: around 124 (the last count that takes pairs) and 2; 4 * 124 * 123 / 2 = 30504 edges
# are the least for 124 of them; stars of 2 and 33 vertices (labels in shared memory), of 34 (4216 vertices: not)
@pytest.mark.parametrize("wmax", [3, 255, 0xFFFFFFFF])
@pytest.mark.parametrize("k,size,m", [(2, 3, 4097), (2, 3, 4096), (123, 2, 40000), (124, 2, 30504), (124, 2, 30503),
                                      (124, 33, 50001), (124, 34, 50001), (125, 33, 50001), (7, 5000, 300001),
                                      (124, 40, 2000003), (60, 60, 1500000)])
def test_pairs_at_their_edges(k, size, m, wmax):
    n, src, dst, w = clusters(k, size, m - k * (size - 1), wmax, 31 * k + size)
    assert src.size == m
    kid, ktot = oracle.kruskal(n, src, dst, w)
    dev = torch.device("cuda", 0)  # base_case=0: small graphs take the rounds too
    for cfg in (dict(base_case=0), dict(base_case=0, variant="filter", filter_min_edges=256, pivot_sample=1024)):
        s = Solver(0, **cfg)
        try:
            for shift in (0, 1):  # at a 16-byte boundary and 4 bytes past one
                t = [torch.zeros(m + shift, dtype=torch.int32, device=dev) for _ in range(3)]
                for x, a in zip(t, (src, dst, w)):
                    x[shift:] = torch.from_numpy(a.view(np.int32)).to(dev)
                ids, tot = s.solve(n, *(x[shift:] for x in t)).to_host()
                assert np.array_equal(ids, kid) and tot == ktot, (cfg, shift)
        finally:
            s.close()
