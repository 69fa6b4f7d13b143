"""The density sweep where particles have more neighbours than fit its stage, up to several hundred,
and where they overrun their lists or have flown far out, against the exact eight-lane sweep."""
import numpy as np
import pytest

from paper_2403_11156_gb300 import scenes, sph

from gpu_util import gpu_ctx

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("squeeze", [0.9, 0.8, 0.6, 0.45])
@pytest.mark.parametrize("cap", [0, 33, 35, 64, 512])
@pytest.mark.parametrize("away", [0, 40])
def test_dense_lists(squeeze, cap, away):
    out = []
    for lanes in (8, 1, 2):
        d = dict(scenes.dam_break_small(seed=4, n=(13, 12, 11), box=0.4), lanes_per_particle=lanes, max_fluid_neighbors=cap)
        x = np.array(d["fluid_x"], np.float32) * np.float32(squeeze)
        if away:      # out of the filter's reach, together in an edge cell
            x[3:3 + away] += np.float32(30.0)
        d["fluid_x"] = x
        d.update(min_iter_density=1, max_iter_density=1, divergence_solve=0, warm_start=scenes.WARM_ZERO)
        g = gpu_ctx(d)
        g.sph_steps(1, 1e-6)
        g.sph_synchronize(raise_on_error=False)
        st = g.sph_get_stats(0)
        out.append((g.sph_read_field(sph.FIELD_NN_FLUID), g.sph_read_field(sph.FIELD_NN_BOUNDARY), g.sph_read_field(sph.FIELD_RHO),
                    g.sph_read_field(sph.FIELD_ALPHA), st["max_fluid_nbrs"], st["max_boundary_nbrs"], st["flags"]))
    assert out[0][4] >= 32
    for b in out[1:]:
        np.testing.assert_array_equal(out[0][0], b[0])
        np.testing.assert_array_equal(out[0][1], b[1])
        # FP32 sums of at most 512 terms in two orders, positive ones for the density; alpha divides
        # by squared sums of as many
        np.testing.assert_allclose(out[0][2], b[2], rtol=512 * 2.0 ** -24)
        np.testing.assert_allclose(out[0][3], b[3], rtol=4 * 512 * 2.0 ** -24)
        assert out[0][4:] == b[4:]
