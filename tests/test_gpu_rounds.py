"""Borůvka rounds in one launch, at the sizes where its tiles, its one-block
finish and its shared-memory minima begin and end; every forest against Kruskal."""
import numpy as np
import pytest
import torch

import oracle
from paper_2302_12199_gb300.mst import Solver

pytestmark = pytest.mark.gpu

# (vertices, edges): one edge; around a tile of 512 and of 2048 edges; around the one-block finish (4096 edges and
# vertices, from the start and after some rounds); more than 4096 components after round 0; several tiles per block
SIZES = [(2, 1), (512, 511), (513, 512), (600, 513), (2048, 2049), (4096, 4096), (4097, 4096), (4096, 4097),
         (5000, 40000), (40000, 39999), (9001, 300001), (700001, 1500003)]


def graph(n, m, wmax, seed):
    """Random edges (self-loops and duplicates among them) over half a random path, so that chains are long."""
    rng = np.random.default_rng(seed)
    src = rng.integers(0, n, m)
    dst = np.where(rng.random(m) < 0.5, np.minimum(src + 1, n - 1), rng.integers(0, n, m))
    w = np.where(rng.random(m) < 0.3, 1 + src % wmax, rng.integers(1, wmax + 1, m))
    return src.astype(np.uint32), dst.astype(np.uint32), w.astype(np.uint32)


@pytest.mark.parametrize("wmax", [255, 0xFFFFFFFF])
@pytest.mark.parametrize("n,m", SIZES)
def test_rounds_at_their_edges(n, m, wmax):
    """Plain Borůvka, and Filter-Borůvka planned and host-driven (whose filter reads the representatives that the
    rounds leave), on arrays at a 16-byte boundary and 4 bytes past one."""
    src, dst, w = graph(n, m, wmax, 17 * n + m)
    kid, ktot = oracle.kruskal(n, src, dst, w)
    dev = torch.device("cuda", 0)
    for cfg in (dict(), dict(variant="filter", filter_min_edges=256, pivot_sample=1024),
                dict(variant="filter", filter_min_edges=256, pivot_sample=1024, filter_plan=0)):
        s = Solver(0, **cfg)
        try:
            for shift in (0, 1):
                t = [torch.zeros(m + shift, dtype=torch.int32, device=dev) for _ in range(3)]
                for x, a in zip(t, (src, dst, w)):
                    x[shift:] = torch.from_numpy(a.view(np.int32)).to(dev)
                ids, tot = s.solve(n, *(x[shift:] for x in t)).to_host()
                assert np.array_equal(ids, kid) and tot == ktot, (cfg, shift)
        finally:
            s.close()
