"""A state written from device arrays (all four in one launch, some of them in two) against the
same state written from the host: the state, the sorted arrays' readable fields, the CFL step
and the next steps bit for bit; and every way of reading it back."""
import numpy as np
import pytest

from paper_2403_11156_gb300 import scenes, sph

from gpu_util import gpu_ctx

pytestmark = pytest.mark.gpu

NAMES = ("x", "v", "kappa_prev", "kappa_v_prev")


@pytest.mark.parametrize("given", [(0, 1, 2, 3), (0, 1), (0,), (1,), (2, 3), (0, 1, 2), ()])
@pytest.mark.parametrize("n", [(1, 1, 1), (5, 3, 17), (8, 8, 4), (257, 1, 1), (9, 11, 13)])
def test_device_write_equals_host_write(n, given):
    import torch
    sizes = [n, (4, 5, 3)]
    descs = [dict(scenes.dam_break_small(seed=3 + k, n=m, box=0.8, warm_start=scenes.WARM_PREVIOUS), cfl=0.4, dt_max=1e-3)
             for k, m in enumerate(sizes)]
    pair = [gpu_ctx(descs), gpu_ctx(descs)]
    nf = len(descs[0]["fluid_x"])
    rng = np.random.default_rng(nf)
    new = [descs[0]["fluid_x"][::-1] + rng.normal(scale=1e-4, size=(nf, 3)), rng.normal(scale=2.0, size=(nf, 3)),
           rng.uniform(0, 1e-7, nf), rng.uniform(0, 1e-4, nf)]
    new = [np.ascontiguousarray(a, dtype=np.float32) for a in new]
    for g in pair:
        g.sph_steps(2)      # the canonical order is no longer the original one
    pair[0].sph_write_state(0, **{NAMES[k]: new[k] for k in given})
    dev = [torch.from_numpy(new[k]).cuda() if k in given else None for k in range(4)]
    torch.cuda.synchronize()
    ptr = [t.data_ptr() if t is not None else None for t in dev]
    assert sph.load().sph_write_state(pair[1].ctx, 0, *ptr, 1) == sph.SPH_OK

    def everything(g, scene):
        fields = [g.sph_read_field(f, scene=scene) for f in (
            sph.FIELD_RHO, sph.FIELD_V_DIV, sph.FIELD_SORTED_ID, sph.FIELD_CELL_KEY, sph.FIELD_KAPPA, sph.FIELD_KAPPA_V,
            sph.FIELD_KAPPA_PREV, sph.FIELD_KAPPA_V_PREV)]
        return fields + list(g.sph_read_state(scene)) + [g.sph_get_stats(scene)["dt_next"]]

    state = pair[1].sph_read_state(0)
    for k in given:
        got = state[k] if k < 2 else pair[1].sph_read_field((sph.FIELD_KAPPA_PREV, sph.FIELD_KAPPA_V_PREV)[k - 2])
        np.testing.assert_array_equal(got, new[k])
    for steps in (0, 1, 1):
        for g in pair:
            g.sph_steps(steps)
        for s in (0, 1):
            for a, b in zip(everything(pair[0], s), everything(pair[1], s)):
                np.testing.assert_array_equal(a, b)
    # the state read into device and host memory, synchronised and only enqueued
    want = pair[1].sph_read_state(0)
    for sync in (True, False):
        out = [torch.empty(a.shape, device="cuda") for a in want]
        pair[1].sph_read_state_device(0, *out, sync=sync)
        host = [np.zeros_like(a) for a in want]
        pair[1].sph_read_state_host(0, *host, sync=sync)
        pair[1].sph_read_wait()
        torch.cuda.synchronize()
        for a, b, c in zip(want, out, host):
            np.testing.assert_array_equal(b.cpu().numpy(), a)
            np.testing.assert_array_equal(c, a)
    part = torch.empty(want[2].shape, device="cuda")
    pair[1].sph_read_state_device(0, rho=part)
    np.testing.assert_array_equal(part.cpu().numpy(), want[2])
