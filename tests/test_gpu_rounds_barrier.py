"""The grid barrier of the one-launch rounds: a wait that runs out ends the call
with MST_ERR_INTERNAL, never with a wrong forest or a pass over unfinished
representatives, and the handle then solves."""
import numpy as np
import pytest
import torch

import oracle
from paper_2302_12199_gb300 import workloads as W
from paper_2302_12199_gb300.mst import MstError, Solver

pytestmark = pytest.mark.gpu

INTERNAL = 6


# plain rounds; rounds whose representatives the filter's passes read next, planned (aligned arrays, and 4 bytes past a
# 16-byte boundary: other filter kernels), host-driven, in two filter passes and with small lists handed back
@pytest.mark.parametrize("shift", [0, 1])
@pytest.mark.parametrize("cfg", [dict(), dict(variant="filter"), dict(variant="filter", filter_plan=0),
                                 dict(variant="filter", filter_split=1), dict(variant="filter", filter_carry=1)])
def test_barrier_that_runs_out_is_an_error(cfg, shift):
    g = W.gnm(1 << 17, 1 << 20, 77)
    kid, ktot = oracle.kruskal(g.n, g.src, g.dst, g.w)
    dev = torch.device("cuda", 0)
    t = [torch.zeros(g.m + shift, dtype=torch.int32, device=dev) for _ in range(3)]
    for x, a in zip(t, (g.src, g.dst, g.w)):
        x[shift:] = torch.from_numpy(a.view(np.int32)).to(dev)
    t = [x[shift:] for x in t]
    s = Solver(0, filter_min_edges=1 << 12, pivot_sample=1 << 12, spin_limit=1, **cfg)
    try:
        statuses = []
        for _ in range(6):
            try:
                ids, tot = s.solve(g.n, *t).to_host()
                assert np.array_equal(ids, kid) and tot == ktot  # OK means exact
                statuses.append(0)
            except MstError as e:
                assert e.status == INTERNAL
                statuses.append(e.status)
        assert INTERNAL in statuses
        s.configure(spin_limit=1 << 21)
        for _ in range(2):
            ids, tot = s.solve(g.n, *t).to_host()
            assert np.array_equal(ids, kid) and tot == ktot
    finally:
        s.close()
