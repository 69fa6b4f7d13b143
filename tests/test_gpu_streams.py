"""Cooperative launches of several streams beside one another and beside other work: two small
contexts (whose solves are one launch each), a grid order and a training on four streams, matrix
products on a fifth; the contexts' states and the order are those of each alone."""
import numpy as np
import pytest

import oracle
from paper_2403_11156_gb300 import scenes, sph, warmstart

from gpu_util import gpu_ctx

pytestmark = pytest.mark.gpu


def test_cooperative_launches_beside_other_work():
    import torch
    descs = [scenes.dam_break_small(seed=2 + k, n=n, box=0.6, warm_start=scenes.WARM_PREVIOUS)
             for k, n in enumerate([(20, 20, 20), (17, 19, 23)])]
    alone = [gpu_ctx(d) for d in descs]
    for g in alone:
        g.sph_steps(25, 4e-4)
        g.sph_synchronize(raise_on_error=False)
    s = [torch.cuda.Stream() for _ in range(5)]
    both = [gpu_ctx(d, stream=q) for d, q in zip(descs, s)]
    rng = np.random.default_rng(1)
    n = 200_003
    x = rng.uniform(0, 2, (n, 3)).astype(np.float32)
    lo, hi, cell = np.zeros(3, np.float32), np.full(3, 2.0, np.float32), np.float32(0.04)
    want = oracle.sort_order(oracle.cell_keys(x, lo, hi, cell))
    xd, order = torch.from_numpy(x).cuda(), torch.empty(n, dtype=torch.int32, device="cuda")
    f, y = torch.randn((20_000, 4), device="cuda"), torch.randn(20_000, device="cuda")
    p = torch.tensor(warmstart.init_params(4), device="cuda")
    adam, hist = torch.zeros(2 * sph.MLP_WEIGHTS, device="cuda"), torch.zeros(2, device="cuda")
    err = torch.zeros(1, dtype=torch.int32, device="cuda")
    a = torch.randn((6000, 6000), device="cuda")
    torch.cuda.synchronize()
    for _ in range(25):
        with torch.cuda.stream(s[4]):
            a @ a
        for g in both:
            g.sph_step(4e-4)
        assert sph.sph_grid_order_noalloc(xd, n, lo, hi, cell, order, None, s[2]) == sph.SPH_OK
        assert sph.sph_mlp_train(f, y, 20_000, p, adam, 2, 4096, 1e-3, 4, hist, err, s[3]) == sph.SPH_OK
    torch.cuda.synchronize()
    assert sph.sph_grid_order_noalloc_status(s[2]) == sph.SPH_OK
    np.testing.assert_array_equal(order.cpu().numpy(), want)
    assert int(err.item()) == 0 and bool(torch.isfinite(p).all())
    for g, h in zip(both, alone):
        assert g.sph_synchronize(raise_on_error=False) != sph.SPH_ETIMEOUT
        for u, v in zip(g.sph_read_state(), h.sph_read_state()):
            np.testing.assert_array_equal(u, v)
