"""The density sweep far from the scene's origin and in domains up to beyond the candidate filter's
range: the same neighbour counts as the exact eight-lane sweep, density within summation order."""
import numpy as np
import pytest

from paper_2403_11156_gb300 import scenes, sph

from gpu_util import gpu_ctx

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("length,shift", [(0.4, 1000.0), (20.0, -500.0), (800.0, 0.0), (8000.0, 100.0), (40_000.0, 0.0)])
@pytest.mark.parametrize("cell", [0.0, 0.0201])
def test_far_and_long(length, shift, cell):
    if cell and length > 10_000:
        pytest.skip("as many cells again twice over")
    out = []
    for lanes in (8, 1, 2):
        d = dict(scenes.dam_break_small(seed=4, n=(13, 11, 12), box=0.4), lanes_per_particle=lanes, cell_size=cell)
        at = np.float32(shift + length - 0.4)     # the far end of the domain
        for k in ("fluid_x", "boundary_x"):
            x = np.array(d[k], np.float64)
            x[:, 0] += at
            d[k] = x.astype(np.float32)
        d["domain_min"] = [shift, 0.0, 0.0]
        d["domain_max"] = [shift + length, 0.4, 0.4]
        d.update(divergence_solve=0, warm_start=scenes.WARM_ZERO, min_iter_density=0, max_iter_density=0)
        g = gpu_ctx(d)
        g.sph_steps(1, 1e-6)
        g.sph_synchronize(raise_on_error=False)
        st = g.sph_get_stats(0)
        out.append((g.sph_read_field(sph.FIELD_NN_FLUID), g.sph_read_field(sph.FIELD_NN_BOUNDARY),
                    g.sph_read_field(sph.FIELD_RHO), st["max_fluid_nbrs"], st["max_boundary_nbrs"], st["flags"]))
        g.close()
    for b in out[1:]:
        np.testing.assert_array_equal(out[0][0], b[0])
        np.testing.assert_array_equal(out[0][1], b[1])
        # FP32 sums of at most 160 positive terms in two orders
        np.testing.assert_allclose(out[0][2], b[2], rtol=1e-5)
        assert out[0][3:] == b[3:]
