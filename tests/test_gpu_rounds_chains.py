"""Pointer jumping of the one-launch rounds on chains around the reach of one and
two passes, and of many; every forest against Kruskal."""
import numpy as np
import pytest
import torch

import oracle
from paper_2302_12199_gb300.mst import Solver

pytestmark = pytest.mark.gpu

STEPS = 32  # parent steps per pass


# lengths around one pass, two passes, the four vertices a thread of a full grid takes at a time; many short chains
SIZES = [(n, chains) for n in (2, STEPS, STEPS + 1, STEPS + 2, STEPS + 3, (STEPS + 1) ** 2, (STEPS + 1) ** 2 + 1,
                               (STEPS + 1) ** 2 + 2, 40000, 700001) for chains in (1, 3, 50) if n * chains < 3_000_000]


@pytest.mark.parametrize("n,chains", SIZES)
def test_chains_at_the_edges_of_a_pass(n, chains):
    """Paths of n vertices with ascending weights, which the first round hooks into one chain each, joined end to end
    by heavier edges."""
    total = n * chains
    src = np.arange(total - 1, dtype=np.uint32)
    pos = np.arange(total - 1) % n
    w = np.where(pos == n - 1, n + 1 + src // n, 1 + pos).astype(np.uint32)
    kid, ktot = oracle.kruskal(total, src, src + 1, w)
    t = [torch.from_numpy(a.view(np.int32)).to("cuda:0") for a in (src, src + 1, w)]
    for cfg in (dict(), dict(variant="filter", filter_min_edges=64, pivot_sample=256),
                dict(variant="filter", filter_min_edges=64, pivot_sample=256, filter_plan=0)):
        s = Solver(0, base_case=0, **cfg)
        try:
            ids, tot = s.solve(total, *t).to_host()
            assert np.array_equal(ids, kid) and tot == ktot, cfg
        finally:
            s.close()
