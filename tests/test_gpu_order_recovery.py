"""The grid order depends on nothing that earlier calls left in its scratch (one that gave up or
overlapped another may leave its histogram and any number of whole barriers): with the rest of the
array overwritten before it, a call and every replay of a captured one give the oracle's order.
And its barrier: blocks that wait in vain give up, a late block too, and the word is whole again
after them.  The array is file-scope, so the source is compiled here beside what reaches it."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

import oracle
from paper_2403_11156_gb300 import build, sph

from gpu_util import gpu_ctx  # noqa: F401  (builds the library)

pytestmark = pytest.mark.gpu

SOURCE = """
#include "sph_noalloc.cu"
extern "C" int fill_scratch(int byte, uint64_t barrier)
{
    void *p = nullptr;
    if (cudaDeviceSynchronize() != cudaSuccess || cudaGetSymbolAddress(&p, g_grid_scratch) != cudaSuccess) return 1;
    if (cudaMemset(p, byte, kScratchBytes) != cudaSuccess) return 2;
    if (cudaMemcpy((char *)p + kOffBar, &barrier, 8, cudaMemcpyHostToDevice) != cudaSuccess) return 3;
    return cudaDeviceSynchronize() != cudaSuccess;
}
// Block `late` comes to the first barrier only after another has given up (or after 2^24 looks).
__global__ void k_late(uint64_t *word, int32_t *error, int32_t *ok, int late)
{
    OrderBarrier bar(word, error);
    if ((int)blockIdx.x == late && threadIdx.x == 0)
        for (int k = 0; k < (1 << 24) && (uint32_t)*(volatile uint64_t *)word == bar.fails; ++k) {}
    const bool came = bar.wait() && bar.wait();
    if (threadIdx.x == 0) ok[blockIdx.x] = came;
    bar.leave(false);
}
extern "C" int run_late(uint64_t *word, int32_t *error, int32_t *ok, int blocks, int late)
{
    void *args[] = {&word, &error, &ok, &late};
    return (int)cudaLaunchCooperativeKernel((const void *)k_late, dim3(blocks), dim3(64), args, 0, 0);
}
// The one-block kernel on control words of the caller's: it needs nothing else that calls share.
extern "C" int run_one(void *ctl, const float *x, int n, int side, float cell, int32_t *order)
{
    Grid g{{-cell, -cell, -cell}, cell, {side, side, side}};
    const int ncell = side * side * side;
    const size_t bytes = sizeof(uint32_t) * (size_t)(kOneBlockMaps + ncell + 1 + n);
    if (cudaFuncSetAttribute(k_na_order_one, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes) != cudaSuccess) return 1;
    k_na_order_one<<<1, kLargeThreads, bytes>>>((Control *)ctl, g, x, n, ncell, nullptr, order);
    return cudaDeviceSynchronize() != cudaSuccess;
}
"""


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    d = tmp_path_factory.mktemp("order")
    src = d / "order.cu"
    src.write_text(SOURCE)
    subprocess.run([build._nvcc(), *build.ARCH, *build.FLAGS, "-shared", "-o", str(d / "order.so"), str(src)], check=True)
    L = ctypes.CDLL(os.fspath(d / "order.so"))
    L.sph_grid_order_noalloc.argtypes = sph.load().sph_grid_order_noalloc.argtypes
    L.sph_grid_order_noalloc_status.argtypes = [ctypes.c_void_p]
    L.fill_scratch.argtypes = [ctypes.c_int, ctypes.c_uint64]
    L.run_one.argtypes = [ctypes.c_void_p] * 2 + [ctypes.c_int] * 2 + [ctypes.c_float] + [ctypes.c_void_p]
    L.run_late.argtypes = [ctypes.c_void_p] * 3 + [ctypes.c_int] * 2
    return L


@pytest.mark.parametrize("byte", [0x00, 0x01, 0x80, 0xA5, 0xFF])
@pytest.mark.parametrize("n,cells,crowd", [(3001, 20, 200), (50_000, 40, 1500), (262_144, 99, 0)])
def test_call_after_anything(lib, n, cells, crowd, byte):
    import torch
    rng = np.random.default_rng(n + byte)
    extent = 0.04 * cells
    f3 = ctypes.c_float * 3
    lo, hi = f3(0.0, 0.0, 0.0), f3(extent, extent, extent)
    x = torch.zeros((n, 3), device="cuda")
    order = torch.full((n,), -1, dtype=torch.int32, device="cuda")
    stream = torch.cuda.Stream()

    def call():
        assert lib.sph_grid_order_noalloc(x.data_ptr(), n, lo, hi, 0.04, order.data_ptr(), None, stream.cuda_stream) == sph.SPH_OK

    def check(enqueue):
        pts = rng.uniform(0, extent, (n, 3)).astype(np.float32)
        pts[:crowd] = np.float32(0.5 * extent)
        x.copy_(torch.from_numpy(pts))
        order.fill_(-1)
        torch.cuda.synchronize()
        # whole barriers (the last before the count starts again among them), calls given up
        assert lib.fill_scratch(byte, int(rng.choice([0, 7 << 48, 0xFFFF << 48])) | byte) == 0
        enqueue()
        assert lib.sph_grid_order_noalloc_status(stream.cuda_stream) == sph.SPH_OK
        want = oracle.sort_order(oracle.cell_keys(pts, np.float32(list(lo)), np.float32(list(hi)), np.float32(0.04)))
        np.testing.assert_array_equal(order.cpu().numpy(), want)

    check(call)
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=stream):
        call()

    def replay():
        with torch.cuda.stream(stream):
            graph.replay()

    for _ in range(2):
        check(replay)
    check(call)


@pytest.mark.parametrize("blocks,late", [(1, -1), (2, -1), (152, -1), (2, 0), (2, 1), (8, 0), (8, 5)])
def test_late_block(lib, blocks, late):
    import torch
    for start in (0, (0xFFFF << 48) | 3):
        word = torch.tensor([start - (1 << 64) if start >> 63 else start], dtype=torch.int64, device="cuda")
        error = torch.zeros(1, dtype=torch.int32, device="cuda")
        ok = torch.full((blocks,), -1, dtype=torch.int32, device="cuda")
        torch.cuda.synchronize()
        assert lib.run_late(word.data_ptr(), error.data_ptr(), ok.data_ptr(), blocks, late) == 0
        torch.cuda.synchronize()
        assert ok.tolist() == [int(late < 0)] * blocks
        assert int(error.item()) == (0 if late < 0 else 5)
        gave_up = blocks if late >= 0 else 0
        assert int(word.item()) % (1 << 64) == (start + (7 << 48) + gave_up) % (1 << 64)


@pytest.mark.parametrize("n,crowds", [(1, 0), (2000, 1), (8192, 126)])
def test_one_block_shares_nothing(lib, n, crowds):
    import torch
    rng = np.random.default_rng(n)
    side, cell = 28, np.float32(0.04)
    extent = float(cell) * (side - 2)
    pts = rng.uniform(0, extent, (n, 3)).astype(np.float32)
    for k in range(crowds):          # 65 points each, beyond what a cell ranks by counting
        pts[65 * k:65 * (k + 1)] = rng.uniform(0, extent, 3)
    pts = pts[rng.permutation(n)]
    ctl = torch.zeros(512, dtype=torch.uint8, device="cuda")
    guard = torch.full((n + 64,), -7, dtype=torch.int32, device="cuda")
    x = torch.from_numpy(pts).cuda()
    torch.cuda.synchronize()
    assert lib.run_one(ctl.data_ptr(), x.data_ptr(), n, side, cell, guard.data_ptr()) == 0
    lo, hi = np.zeros(3, np.float32), np.full(3, extent, np.float32)
    np.testing.assert_array_equal(guard[:n].cpu().numpy(), oracle.sort_order(oracle.cell_keys(pts, lo, hi, cell)))
    assert bool((guard[n:] == -7).all())
