"""Planned Filter-Borůvka where the light list's length lies at the bound that
decides whether it is partitioned again: on either side of what was expected, the
plan holds and the forest is Kruskal's."""
import numpy as np
import pytest
import torch

import oracle
from paper_2302_12199_gb300.mst import Solver

pytestmark = pytest.mark.gpu


# the expected light share is m / 8 edges, the bound n (average degree 2): below it, at it, above it by less and by more
# than the sample strays
@pytest.mark.parametrize("wmax", [255, 0xFFFFFFFF])
@pytest.mark.parametrize("excess", [-400, -20, 0, 1, 20, 400])
def test_plan_holds_at_the_sparsity_bound(excess, wmax):
    n = 1 << 14
    m = 8 * (n + excess)
    for seed in range(4):
        rng = np.random.default_rng(seed)
        src, dst = (rng.integers(0, n, m).astype(np.uint32) for _ in range(2))
        w = rng.integers(1, wmax, m, endpoint=True).astype(np.uint32)
        kid, ktot = oracle.kruskal(n, src, dst, w)
        t = [torch.from_numpy(a.view(np.int32)).to("cuda:0") for a in (src, dst, w)]
        s = Solver(0, variant="filter", pivot_quantile=0.125, filter_min_edges=256, filter_max_avg_degree=2.0,
                   pivot_sample=1024, seed=seed)
        try:
            for _ in range(2):
                ids, tot = s.solve(n, *t).to_host()
                assert np.array_equal(ids, kid) and tot == ktot
            hc = s.host_counters()
            assert hc["planned"] == 2 and hc["plan_fallbacks"] == 0, hc
        finally:
            s.close()
