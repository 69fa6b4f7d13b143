"""The surface of a large grid, whose blocks take tiles of eight cubes a thread, against that of its
slabs, which are small enough for one cube a thread: the same triangles, bit for bit and in order
(spacing and origins are powers of two, so a slab's coordinates are the grid's).  And small grids do
not take as long as a few blocks would."""
import ctypes

import numpy as np
import pytest

from paper_2403_11156_gb300 import sph

from gpu_util import gpu_ctx  # noqa: F401  (builds the library)

pytestmark = pytest.mark.gpu


def _mesh(field, z0, cap):
    import torch
    dims = (ctypes.c_int32 * 3)(field.shape[2], field.shape[1], field.shape[0])
    out = torch.full((cap, 3, 3), -9.0, device="cuda")
    n = ctypes.c_int64()
    st = sph.load().sph_surface_mesh(field.data_ptr(), dims, (ctypes.c_float * 3)(-2.0, 1.0, z0 * 0.25), 0.25, 0.5,
                                     out.data_ptr(), cap, ctypes.byref(n), torch.cuda.current_stream().cuda_stream)
    assert st in (sph.SPH_OK, sph.SPH_EOVERFLOW) and (st == sph.SPH_OK) == (n.value <= cap)
    return out[:n.value], n.value


@pytest.mark.parametrize("dims", [(130, 121, 111), (2049, 29, 30), (5, 641, 650)])
@pytest.mark.parametrize("noise", [0.0, 0.05])
def test_large_grid_equals_its_slabs(dims, noise):
    import torch
    nx, ny, nz = dims
    assert (nx - 1) * (ny - 1) * (nz - 1) >= 5 * 152 * 2048
    g = torch.Generator(device="cuda").manual_seed(nx)
    ax = [torch.linspace(-1, 1, m, device="cuda") for m in (nz, ny, nx)]
    z, y, x = torch.meshgrid(*ax, indexing="ij")
    f = (1.2 - (x * x + y * y + z * z).sqrt() + noise * torch.randn((nz, ny, nx), generator=g, device="cuda")).contiguous()
    whole, n = _mesh(f, 0, 4_000_000)
    parts, step = [], 23
    for k in range(0, nz - 1, step):
        parts.append(_mesh(f[k:k + step + 1].contiguous(), k, 2_000_000)[0])
    parts = torch.cat(parts)
    assert n == len(parts) and n > 1000
    assert torch.equal(whole, parts)
    # a buffer too small: what fits, nothing beyond
    cut, m = _mesh(f, 0, n // 2)
    assert m == n and torch.equal(cut, whole[:n // 2])


def test_small_grid_is_not_slow():
    import torch
    from torch.profiler import ProfilerActivity, profile
    us = []
    for m in (101, 17, 101):      # (a process's first profile may come out empty)
        f = torch.rand((m, m, m), device="cuda")
        for _ in range(2):
            n = _mesh(f, 0, 8_000_000)[1]
        with profile(activities=[ProfilerActivity.CUDA]) as p:
            for _ in range(5):
                _mesh(f, 0, 8_000_000)
        us.append(sum(e.self_device_time_total for e in p.key_averages() if "k_mt_emit" in e.key) / 5)
        assert n > 1000
    # 4,096 cubes against 1,000,000, all crossed
    assert 0.0 < us[1] < us[2] / 5, us
