"""The grid order without allocation at the edges of its two kernels (one block up to 8,192
points and 24,576 cells, all blocks beyond), with crowded cells, against the oracle; call after
call on one scratch array."""
import numpy as np
import pytest

import oracle
from paper_2403_11156_gb300 import sph

from gpu_util import gpu_ctx  # noqa: F401  (builds the library)

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,cells,crowd", [
    (1, 3, 0), (31, 1, 0), (1024, 10, 65), (8191, 20, 0), (8192, 20, 700), (8193, 20, 700), (3000, 26, 0), (3000, 27, 0),
    (3000, 28, 2000), (5000, 2, 0), (1025, 99, 0), (100_001, 60, 1500), (262_144, 99, 0), (262_144, 14, 0)])
def test_order(n, cells, crowd):
    import torch
    rng = np.random.default_rng(n + cells)
    extent = 0.04 * cells
    x = rng.uniform(-0.02, extent + 0.02, (n, 3)).astype(np.float32)   # some outside: clamped
    if crowd:
        x[rng.permutation(n)[:crowd]] = np.float32(0.5 * extent)
    lo, hi = np.zeros(3, np.float32), np.full(3, extent, np.float32)
    keys_o = oracle.cell_keys(x, lo, hi, np.float32(0.04))
    order_o = oracle.sort_order(keys_o)
    xd = torch.from_numpy(x).cuda()
    for keys_too in (True, False, True):
        order = torch.full((n,), -1, dtype=torch.int32, device="cuda")
        keys = torch.zeros(n, dtype=torch.int32, device="cuda") if keys_too else None
        assert sph.sph_grid_order_noalloc(xd, n, lo, hi, np.float32(0.04), order, keys) == sph.SPH_OK
        assert sph.sph_grid_order_noalloc_status(torch.cuda.current_stream()) == sph.SPH_OK
        np.testing.assert_array_equal(order.cpu().numpy(), order_o)
        if keys_too:
            np.testing.assert_array_equal(keys.cpu().numpy().view(np.uint32), keys_o)


@pytest.mark.parametrize("n,cells", [(3001, 20), (50_000, 40)])
def test_order_under_capture(n, cells):
    """Enqueued into another component's graph capture, and replayed on other points."""
    import torch
    rng = np.random.default_rng(n)
    extent = 0.04 * cells
    lo, hi = np.zeros(3, np.float32), np.full(3, extent, np.float32)
    x = torch.zeros((n, 3), device="cuda")
    order = torch.full((n,), -1, dtype=torch.int32, device="cuda")
    stream = torch.cuda.Stream()
    with torch.cuda.stream(stream):
        assert sph.sph_grid_order_noalloc(x, n, lo, hi, np.float32(0.04), order, None, stream) == sph.SPH_OK
    stream.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=stream):
        assert sph.sph_grid_order_noalloc(x, n, lo, hi, np.float32(0.04), order, None, stream) == sph.SPH_OK
    for _ in range(3):
        pts = rng.uniform(0, extent, (n, 3)).astype(np.float32)
        x.copy_(torch.from_numpy(pts))
        torch.cuda.synchronize()
        graph.replay()
        torch.cuda.synchronize()
        want = oracle.sort_order(oracle.cell_keys(pts, lo, hi, np.float32(0.04)))
        np.testing.assert_array_equal(order.cpu().numpy(), want)
