"""The tiled field kernel against the general one, bit for bit at the nodes both have, and the
one-pass surface on noise over ragged grids against the oracle."""
import numpy as np
import pytest

from oracle import postprocess as post
from paper_2403_11156_gb300 import scenes, sph

from gpu_util import gpu_ctx

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("cell,origin,dims", [
    (0.0, (0.0, 0.0, 0.0), (41, 41, 41)),
    (0.0, (-0.013, 0.007, -0.3), (57, 33, 81)),      # nodes outside the domain, ragged tiles
    (0.0201, (0.0, 0.0, 0.0), (40, 37, 45)),         # cells of h/2: a stencil of 5 x 5 rows
    (0.0, (0.1, 0.1, 0.02), (1, 1, 1)),
    (0.0, (0.05, 0.05, 0.0), (5, 9, 65)),
])
@pytest.mark.parametrize("lists", [0, 2])            # 2: lists too short to serve as scratch
def test_tiles_equal_the_general_kernel(cell, origin, dims, lists):
    d = scenes.dam_break_small(seed=9, n=(9, 11, 13), box=0.4)
    d = dict(d, cell_size=cell, max_fluid_neighbors=lists)
    g = gpu_ctx(d)
    if not lists:
        g.sph_steps(3)
    h = 4.0 * d["radius"]
    s = float(np.float32(h) * np.float32(0.2421875))  # 4 s is exact and above the tiles' limit
    fine = g.sph_surface_field(origin, s, dims).cpu().numpy()
    coarse = g.sph_surface_field(origin, 4.0 * s, [(n + 3) // 4 for n in dims]).cpu().numpy()
    np.testing.assert_array_equal(fine[::4, ::4, ::4], coarse)
    assert dims[0] * dims[1] * dims[2] < 100 or fine.max() > 0.5


@pytest.mark.parametrize("dims", [(2, 2, 2), (3, 5, 131), (258, 2, 3), (2, 300, 2), (17, 16, 9)])
def test_surface_of_noise(dims):
    import ctypes
    import torch
    rng = np.random.default_rng(sum(dims))
    f = rng.random(dims[::-1]).astype(np.float32)
    f[f > 0.97] = 0.5                                # corners exactly at the iso-level
    ref = post.marching_tetrahedra(f, (0.1, -0.2, 0.3), 0.25, 0.5)
    field = torch.from_numpy(f).cuda()
    out = torch.full((len(ref) + 2, 3, 3), 9.0, device="cuda")
    n = ctypes.c_int64()
    args = ((ctypes.c_int32 * 3)(*dims), (ctypes.c_float * 3)(0.1, -0.2, 0.3), 0.25, 0.5)
    run = lambda t, cap: sph.load().sph_surface_mesh(  # noqa: E731
        field.data_ptr(), *args, t, cap, ctypes.byref(n), torch.cuda.current_stream().cuda_stream)
    assert run(out.data_ptr(), len(ref)) == sph.SPH_OK and n.value == len(ref)
    got = out[:len(ref)].cpu().numpy()
    # slivers may turn over with the rounding of the coordinates (orientation on smooth fields:
    # test_gpu_post): the last two vertices in either order, almost all in the oracle's
    turned = np.abs(got - ref).max(axis=(1, 2)) > np.abs(got[:, [0, 2, 1]] - ref).max(axis=(1, 2))
    assert turned.mean() < 0.01
    got[turned] = got[turned][:, [0, 2, 1]]
    # an FP32 vertex: two roundings of its coordinate (up to 75) and of the cut along the edge
    np.testing.assert_allclose(got, ref, rtol=2.0 ** -22, atol=1e-6)
    assert bool((out[len(ref):] == 9.0).all())
    # too small a buffer: what fits, the full count, an error
    part = torch.full((len(ref) + 2, 3, 3), 9.0, device="cuda")
    cap = len(ref) // 2
    assert run(part.data_ptr(), cap) == sph.SPH_EOVERFLOW and n.value == len(ref)
    assert torch.equal(part[:cap], out[:cap]) and bool((part[cap:] == 9.0).all())
    assert run(None, 0) == sph.SPH_EOVERFLOW and n.value == len(ref)
