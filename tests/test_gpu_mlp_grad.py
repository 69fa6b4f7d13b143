"""The network's gradient kernel at the edges of its 128-sample tiles, over several tiles a
CTA and into a gradient buffer that is not 16-byte aligned, against the oracle's FP64 one."""
import numpy as np
import pytest

import oracle
from paper_2403_11156_gb300 import sph

from gpu_util import gpu_ctx  # noqa: F401  (builds the library)

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,offset", [(1, 0), (127, 0), (128, 1), (129, 2), (3 * 128 - 1, 0), (128 * 304 + 1, 0),
                                      (128 * 650 + 77, 3)])
def test_gradient_tiles(n, offset):
    import torch
    rng = np.random.default_rng(n)
    p = np.zeros(sph.MLP_PARAMS, np.float32)
    p[:sph.MLP_WEIGHTS] = rng.normal(scale=0.3, size=sph.MLP_WEIGHTS)
    p[sph.MLP_WEIGHTS + 4:sph.MLP_WEIGHTS + 8] = 1.0
    p[-1] = 1.0
    f = rng.normal(size=(n, 4)).astype(np.float32)
    t = (rng.normal(size=n) + 8.0).astype(np.float32)   # labels off the outputs: no cancellation in dy
    dev = lambda a: torch.tensor(a, device="cuda")  # noqa: E731
    buf = torch.full((sph.MLP_WEIGHTS + 8,), 7.0, device="cuda")
    g = buf[offset:offset + sph.MLP_WEIGHTS]
    loss = torch.zeros(1, dtype=torch.float64, device="cuda")
    err = torch.zeros(1, dtype=torch.int32, device="cuda")
    assert sph.sph_mlp_grad(dev(p), dev(f), dev(t), n, g, loss, err) == sph.SPH_OK
    torch.cuda.synchronize()
    assert int(err.item()) == 0
    ref_loss, ref = oracle.mlp_loss_grad(p.astype(np.float64), f.astype(np.float64), t.astype(np.float64))
    # BF16 operands (2^-9 each) through three products: normwise 2e-2, as in test_gpu_mlp
    assert float(loss.item()) / n == pytest.approx(ref_loss, rel=2e-2)
    got = g.cpu().numpy().astype(np.float64)
    for lo, hi in [(0, 4545), (0, 256), (256, 320), (320, 4416), (4416, 4480), (4480, 4544), (4544, 4545)]:
        assert np.linalg.norm(got[lo:hi] - ref[lo:hi]) <= 2e-2 * np.linalg.norm(ref[lo:hi])
    rest = torch.cat([buf[:offset], buf[offset + sph.MLP_WEIGHTS:]])
    assert bool((rest == 7.0).all())


@pytest.mark.parametrize("n", [1, 128, 129, 128 * 152 * 7 + 5])
def test_forward_non_finite_rows(n):
    """A NaN or infinite feature gives NaN in its own row and changes no other."""
    import torch
    rng = np.random.default_rng(n)
    p = np.zeros(sph.MLP_PARAMS, np.float32)
    p[:sph.MLP_WEIGHTS] = rng.normal(scale=0.3, size=sph.MLP_WEIGHTS)
    f = torch.tensor(rng.normal(size=(n, 4)).astype(np.float32), device="cuda")
    dp = torch.tensor(p, device="cuda")
    err = torch.zeros(1, dtype=torch.int32, device="cuda")
    y = [torch.empty(n, device="cuda") for _ in range(2)]
    assert sph.sph_mlp_forward(dp, f, n, y[0], err) == sph.SPH_OK
    bad = sorted({0, n // 2, n - 1})
    for k, i in enumerate(bad):
        f[i, k % 4] = [float("nan"), float("inf"), float("-inf")][k]
    assert sph.sph_mlp_forward(dp, f, n, y[1], err) == sph.SPH_OK
    torch.cuda.synchronize()
    assert int(err.item()) == 0
    keep = torch.ones(n, dtype=torch.bool, device="cuda")
    keep[bad] = False
    assert bool(torch.isnan(y[1][~keep]).all())
    assert torch.equal(y[0][keep], y[1][keep])


@pytest.mark.parametrize("n,batch", [(2, 1), (129, 128), (300, 127), (1000, 5000), (20_003, 4096), (128 * 310 + 1, 128 * 305)])
def test_epochs_cover_every_sample_once(n, batch):
    """With a vanishing learning rate every epoch's mean loss is that of the initial network
    over all (standardised) samples, whatever the batches."""
    import torch
    rng = np.random.default_rng(n)
    p = np.zeros(sph.MLP_PARAMS, np.float32)
    p[:sph.MLP_WEIGHTS] = rng.normal(scale=0.3, size=sph.MLP_WEIGHTS)
    f = (rng.normal(size=(n, 4)) * [1.0, 3.0, 0.5, 2.0] + 1.0).astype(np.float32)
    t = (rng.normal(size=n) * 2.0 + 5.0).astype(np.float32)
    dev = lambda a: torch.tensor(a, device="cuda")  # noqa: E731
    dp, adam = dev(p), torch.zeros(2 * sph.MLP_WEIGHTS, device="cuda")
    hist, err = torch.zeros(3, device="cuda"), torch.zeros(1, dtype=torch.int32, device="cuda")
    assert sph.sph_mlp_train(dev(f), dev(t), n, dp, adam, 3, batch, 1e-20, 5, hist, err) == sph.SPH_OK
    torch.cuda.synchronize()
    assert int(err.item()) == 0
    std = lambda a: (a - a.mean(0)) / a.std(0)  # noqa: E731
    ref, _ = oracle.mlp_loss_grad(p.astype(np.float64), std(f.astype(np.float64)), std(t.astype(np.float64)))
    # BF16 operands: 2e-2, as for the gradient's loss
    np.testing.assert_allclose(hist.cpu().numpy(), ref, rtol=2e-2)
    np.testing.assert_array_equal(dp.cpu().numpy()[:sph.MLP_WEIGHTS], p[:sph.MLP_WEIGHTS])
