"""Launches that the runtime refuses (a full device, an attribute that could not
be set): the call takes the general path and gives the same forest.  The library
is linked a second time here with a stand-in for the launch calls, which returns
an error for the kernels that a test names and passes the others on."""
import concurrent.futures as cf
import ctypes
import os
import subprocess

import numpy as np
import pytest
import torch

import oracle
from paper_2302_12199_gb300 import build as B
from paper_2302_12199_gb300 import mst
from paper_2302_12199_gb300 import workloads as W

pytestmark = pytest.mark.gpu

STAND_IN = r"""
#include <cstring>
#include <cuda_runtime.h>
static const char *g_name = nullptr;  // refuse the kernels whose name holds this
static int g_refused = 0;
extern "C" void refuse(const char *name) { g_name = name; g_refused = 0; }
extern "C" int refused() { return g_refused; }
static bool no(const void *f) {
  const char *name = nullptr;
  if (!g_name || cudaFuncGetName(&name, f) != cudaSuccess || !std::strstr(name, g_name)) return false;
  ++g_refused;
  return true;
}
extern "C" {
cudaError_t __real_cudaLaunchKernel(const void *, dim3, dim3, void **, size_t, cudaStream_t);
cudaError_t __wrap_cudaLaunchKernel(const void *f, dim3 g, dim3 b, void **a, size_t m, cudaStream_t s) {
  return no(f) ? cudaErrorLaunchOutOfResources : __real_cudaLaunchKernel(f, g, b, a, m, s);
}
cudaError_t __real_cudaLaunchCooperativeKernel(const void *, dim3, dim3, void **, size_t, cudaStream_t);
cudaError_t __wrap_cudaLaunchCooperativeKernel(const void *f, dim3 g, dim3 b, void **a, size_t m, cudaStream_t s) {
  return no(f) ? cudaErrorCooperativeLaunchTooLarge : __real_cudaLaunchCooperativeKernel(f, g, b, a, m, s);
}
}
"""


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    d = tmp_path_factory.mktemp("refused")
    (d / "stand_in.cu").write_text(STAND_IN)
    srcs = B.sources() + [str(d / "stand_in.cu")]

    def compile_one(src):
        obj = str(d / (os.path.basename(src) + ".o"))
        subprocess.run([B.nvcc(), "-c", src, "-o", obj] + B.ARCH + B.NVCC_FLAGS, check=True)
        return obj
    with cf.ThreadPoolExecutor(len(srcs)) as ex:
        objs = list(ex.map(compile_one, srcs))
    so = str(d / "librefused.so")
    wrap = [x for f in ("cudaLaunchKernel", "cudaLaunchCooperativeKernel") for x in ("-Xlinker", "--wrap=" + f)]
    subprocess.run([B.nvcc(), "-shared", "-o", so] + B.ARCH + wrap + objs, check=True)
    so = ctypes.CDLL(so)
    for name, (res, args) in mst._SIGNATURES.items():
        getattr(so, name).restype, getattr(so, name).argtypes = res, args
    so.refuse.argtypes = [ctypes.c_char_p]
    yield so
    so.refuse(None)


def to_dev(g):
    return [torch.from_numpy(a.view(np.int32)).to("cuda:0") for a in (g.src, g.dst, g.w)]


def test_refused_block_launch_of_a_small_graph(lib, monkeypatch):
    monkeypatch.setattr(mst, "_lib", lib)
    g = W.gnm(3000, 20000, 5)
    kid, ktot = oracle.kruskal(g.n, g.src, g.dst, g.w)
    s = mst.Solver(0)
    try:
        for name, hits in ((b"block_single", 1), (None, 0)):
            lib.refuse(name)
            ids, tot = s.solve(g.n, *to_dev(g)).to_host()
            assert np.array_equal(ids, kid) and tot == ktot and lib.refused() == hits
    finally:
        lib.refuse(None)
        s.close()


# every kind of block, and one of the three (its name ends by the block's threads)
@pytest.mark.parametrize("name", [b"block_batch", b"block_batch_kernelILi256", b"block_batch_kernelILi512",
                                  b"block_batch_kernelILi1024"])
@pytest.mark.parametrize("copies", [1, 60])  # in one stream, and side by side in three
def test_refused_block_launch_in_a_batch(lib, monkeypatch, name, copies):
    monkeypatch.setattr(mst, "_lib", lib)
    graphs = [W.gnm(n, 2 * n, 7 + n) for n in (500, 14000, 30000)] * copies
    off = np.cumsum([0] + [g.m for g in graphs]).astype(np.uint64)
    t = [torch.from_numpy(np.concatenate([getattr(g, k) for g in graphs]).view(np.int32)).to("cuda:0")
         for k in ("src", "dst", "w")]
    want = [oracle.kruskal(g.n, g.src, g.dst, g.w) for g in graphs[:3]]
    s = mst.Solver(0)
    try:
        for refuse in (name, None):
            lib.refuse(refuse)
            ids, moff, tot = s.solve_batched(np.array([g.n for g in graphs], np.uint32), off, *t)
            ids, moff, tot = ids.cpu().numpy().view(np.uint32), moff.cpu().numpy(), tot.cpu().numpy()
            for i in range(len(graphs)):
                assert np.array_equal(ids[moff[i]:moff[i + 1]], want[i % 3][0]) and tot[i] == want[i % 3][1], i
    finally:
        lib.refuse(None)
        s.close()


# plain rounds, and Filter-Borůvka planned with light lists on either side of the sparsity bound, several levels deep,
# with packed and unpacked keys
@pytest.mark.parametrize("cfg", [dict(), dict(variant="filter"), dict(variant="filter", filter_max_avg_degree=4.0),
                                 dict(variant="filter", pivot_quantile=0.5), dict(variant="filter", filter_plan=0)])
@pytest.mark.parametrize("wmax", [255, 0xFFFFFFFF])
def test_refused_rounds(lib, monkeypatch, cfg, wmax):
    monkeypatch.setattr(mst, "_lib", lib)
    g = W.gnm(1 << 14, 1 << 18, 9)
    w = np.random.default_rng(4).integers(1, wmax, g.m, endpoint=True).astype(np.uint32)
    kid, ktot = oracle.kruskal(g.n, g.src, g.dst, w)
    t = to_dev(W.Graph(g.n, g.src, g.dst, w))
    s = mst.Solver(0, filter_min_edges=1 << 10, pivot_sample=1 << 12, **cfg)
    try:
        for name in (b"rounds_kernel", None, b"rounds_kernel"):
            lib.refuse(name)
            ids, tot = s.solve(g.n, *t).to_host()
            assert np.array_equal(ids, kid) and tot == ktot
            assert (lib.refused() > 0) == (name is not None)
    finally:
        lib.refuse(None)
        s.close()
