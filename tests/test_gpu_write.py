"""A written state: the next step's CFL step from the largest speed in any block, values that
are not given kept (in original particle order), and the enqueued and synchronous reads."""
import numpy as np
import pytest

from paper_2403_11156_gb300 import scenes

from gpu_util import gpu_ctx

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,at", [((1, 1, 1), 0), ((5, 3, 17), 254), ((8, 8, 4), 255), ((9, 11, 13), 1000)])
def test_written_state(n, at):
    d = scenes.dam_break_small(seed=3, n=n, box=0.8)
    d = dict(d, cfl=0.4, dt_max=1e-2)
    g = gpu_ctx(d)
    g.sph_steps(2)   # the canonical order is no longer the original one
    before = g.sph_read_state()
    nf = len(d["fluid_x"])
    rng = np.random.default_rng(nf)
    v = rng.normal(scale=0.1, size=(nf, 3)).astype(np.float32)
    v[at] = [3.0, -4.0, 12.0]
    g.sph_write_state(0, v=v)
    x, vel = g.sph_read_state()[:2]
    np.testing.assert_array_equal(vel, v)
    np.testing.assert_array_equal(x, before[0])
    want = np.float32(np.float32(d["cfl"]) * np.float32(2.0 * d["radius"]) / np.float32(13.0))
    assert g.sph_get_stats(0)["dt_next"] == pytest.approx(float(want), rel=1e-6)
    g.sph_write_state(0, x=before[0][::-1].copy(), v=np.zeros_like(v))
    x, vel = g.sph_read_state()[:2]
    np.testing.assert_array_equal(x, before[0][::-1])
    assert not vel.any()
    assert g.sph_get_stats(0)["dt_next"] == pytest.approx(float(np.float32(d["dt_max"])), rel=1e-6)
