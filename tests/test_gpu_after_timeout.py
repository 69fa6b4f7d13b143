"""After a bounded device wait gave up, what is queued behind it does not wait as long again: further
launches on the same grid barrier (the one-launch solves of a context's queued steps), and the
epochs of a training, which return at once."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

from paper_2403_11156_gb300 import build, sph

from gpu_util import gpu_ctx  # noqa: F401  (builds the library)

pytestmark = pytest.mark.gpu


SOURCE = """
#include "sph_mlp_train.cu"
// A barrier that block 0 does not come to.
__global__ void k_wait(GridBar *bar, int32_t *error)
{
    if (blockIdx.x == 0) return;
    uint32_t phase = *reinterpret_cast<volatile uint32_t *>(&bar->gen);
    grid_barrier(bar, error, phase);
}
extern "C" int run_wait(GridBar *bar, int32_t *error, int blocks, float *ms)
{
    cudaEvent_t e[2];
    for (auto &x : e) cudaEventCreate(&x);
    void *args[] = {&bar, &error};
    cudaEventRecord(e[0]);
    if (cudaLaunchCooperativeKernel((const void *)k_wait, dim3(blocks), dim3(kBlock), args, 0, 0) != cudaSuccess) return 2;
    cudaEventRecord(e[1]);
    if (cudaDeviceSynchronize() != cudaSuccess) return 1;
    cudaEventElapsedTime(ms, e[0], e[1]);
    for (auto &x : e) cudaEventDestroy(x);
    return 0;
}
// One epoch over n <= 128 samples with the barrier's state given.
extern "C" int run_epoch(float *w, float *mv, float *grad, const float *F, const float *T, int64_t n, double *acc,
                         float *history, void *sync, int *err)
{
    float *m = mv, *v = mv + kNW;
    const float4 *f = (const float4 *)F;
    int64_t batch = n, step = 0;
    uint64_t a = 1, c = 0;
    AdamArgs h{1e-3f, 0.9f, 0.999f, 1e-8f};
    EpochSync *es = (EpochSync *)sync;
    if (set_attr() != cudaSuccess) return 1;
    void *args[] = {&w, &m, &v, &grad, &f, &T, &n, &batch, &a, &c, &step, &h, &acc, &history, &es, &err};
    if (cudaLaunchCooperativeKernel((const void *)k_mlp_epoch, dim3(1), dim3(kThreads), args, kSmem, 0) != cudaSuccess) return 2;
    return cudaDeviceSynchronize() != cudaSuccess;
}
"""


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    d = tmp_path_factory.mktemp("epoch")
    src = d / "epoch.cu"
    src.write_text(SOURCE)
    subprocess.run([build._nvcc(), *build.ARCH, *build.FLAGS, "-shared", "-o", str(d / "epoch.so"), str(src)], check=True)
    L = ctypes.CDLL(os.fspath(d / "epoch.so"))
    L.run_epoch.argtypes = [ctypes.c_void_p] * 5 + [ctypes.c_int64] + [ctypes.c_void_p] * 4
    L.run_wait.argtypes = [ctypes.c_void_p] * 2 + [ctypes.c_int, ctypes.POINTER(ctypes.c_float)]
    return L


def test_launches_on_a_failed_barrier(lib):
    import torch
    bar, error = torch.zeros(2, dtype=torch.int32, device="cuda"), torch.zeros(1, dtype=torch.int32, device="cuda")
    torch.cuda.synchronize()
    times = []
    for _ in range(5):
        ms = ctypes.c_float()
        assert lib.run_wait(bar.data_ptr(), error.data_ptr(), 152, ctypes.byref(ms)) == 0
        times.append(ms.value)
        assert int(error.item()) == 5
    # 2^21 looks the first time, at most 2^10 afterwards
    assert max(times[1:]) < times[0] / 20, times


def test_epochs_after_a_failed_one(lib):
    import torch
    rng = np.random.default_rng(1)
    n = 100
    p = torch.tensor(rng.normal(scale=0.3, size=sph.MLP_PARAMS).astype(np.float32), device="cuda")
    f, t = torch.randn((n, 4), device="cuda"), torch.randn(n, device="cuda")
    for failed in (0, 1):
        w = p.clone()
        mv, grad = torch.zeros(2 * sph.MLP_WEIGHTS, device="cuda"), torch.zeros(sph.MLP_WEIGHTS, device="cuda")
        acc, hist = torch.zeros(12, dtype=torch.float64, device="cuda"), torch.full((1,), -1.0, device="cuda")
        # a barrier that an earlier epoch left half full, and the mark of its failure
        sync = torch.tensor([failed * 7, failed * 3, failed, 0], dtype=torch.int32, device="cuda")
        err = torch.zeros(1, dtype=torch.int32, device="cuda")
        torch.cuda.synchronize()
        args = (w, mv, grad, f, t, n, acc, hist, sync, err)
        assert lib.run_epoch(*(a.data_ptr() if torch.is_tensor(a) else a for a in args)) == 0
        assert torch.equal(w, p) == bool(failed)
        assert (float(hist.item()) == -1.0) == bool(failed)
        assert int(err.item()) == 5 * failed
