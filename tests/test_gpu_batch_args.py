"""Arrays of a batch that are not 4-byte aligned are refused before any pass reads
them, whichever way the batch would be solved."""
import ctypes

import numpy as np
import pytest
import torch

from paper_2302_12199_gb300 import mst
from paper_2302_12199_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("base_case", [0, 1])  # the union, and a block per graph
@pytest.mark.parametrize("which", range(4))    # src, dst, w, ids
@pytest.mark.parametrize("shift", [1, 2])
def test_unaligned_batch_arrays_are_refused(base_case, which, shift):
    dev = torch.device("cuda", 0)
    g = W.gnm(500, 3000, 3)
    t = [torch.zeros(4 * g.m + 8, dtype=torch.uint8, device=dev) for _ in range(4)]
    for x, a in zip(t, (g.src, g.dst, g.w)):
        x[:4 * g.m] = torch.from_numpy(a.view(np.uint8)).to(dev)
    n = torch.tensor([g.n], dtype=torch.int32, device=dev)
    off = torch.tensor([0, g.m], dtype=torch.int64, device=dev)
    moff, tot = (torch.zeros(2, dtype=torch.int64, device=dev) for _ in range(2))
    ptr = [x.data_ptr() + (shift if k == which else 0) for k, x in enumerate(t)]
    s = mst.Solver(0, base_case=base_case)
    try:
        st = s.lib.mst_solve_batched(s.h, 1, n.data_ptr(), off.data_ptr(), *ptr, moff.data_ptr(), tot.data_ptr(),
                                     ctypes.c_void_p(torch.cuda.current_stream().cuda_stream))
        assert st == 1  # MST_ERR_INVALID_ARG
        ids, moff, tot = s.solve_batched(np.array([g.n], np.uint32), np.array([0, g.m], np.uint64),
                                         *(x[:4 * g.m].view(torch.int32) for x in t[:3]))
        assert int(moff[1]) > 0 and int(tot[0]) > 0
    finally:
        s.close()
