"""One-launch rounds that end because hooking leaves a single component, in the
first round or a later one, with and without representatives to hand on; every
forest against Kruskal."""
import numpy as np
import pytest
import torch

import oracle
from paper_2302_12199_gb300.mst import Solver

pytestmark = pytest.mark.gpu


# (vertices, edges): two vertices and their parallel edges; stars whose list is just within and past the one-block
# finish, a tile of the whole grid, and beyond it; `halves`: two stars, which one round leaves and the next joins
@pytest.mark.parametrize("n,m", [(2, 1), (2, 5000), (300, 4096), (300, 4097), (4096, 70000), (5000, 70000),
                                 (50000, 700001), (400, 1500000)])
@pytest.mark.parametrize("halves", [False, True])
def test_rounds_that_end_in_one_component(n, m, halves):
    rng = np.random.default_rng(n + m)
    leaf = np.minimum(np.arange(m) % n, n - 1)
    hub = np.where(leaf < n // 2, 0, n // 2) if halves else np.zeros(m, np.int64)
    w = rng.integers(2, 1000, m)
    if halves:  # the lightest edges stay in a half; the last edge joins them
        leaf[-1], hub[-1], w[-1] = n - 1, 0, 5000
    src, dst, w = (a.astype(np.uint32) for a in (hub, leaf, w))
    kid, ktot = oracle.kruskal(n, src, dst, w)
    t = [torch.from_numpy(a.view(np.int32)).to("cuda:0") for a in (src, dst, w)]
    for cfg in (dict(), dict(variant="filter", filter_min_edges=64, pivot_sample=256),
                dict(variant="filter", filter_min_edges=64, pivot_sample=256, filter_plan=0)):
        s = Solver(0, base_case=0, **cfg)
        try:
            for _ in range(2):
                ids, tot = s.solve(n, *t).to_host()
                assert np.array_equal(ids, kid) and tot == ktot, cfg
        finally:
            s.close()
