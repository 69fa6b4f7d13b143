"""The eight-lane density sweep with 32, 16 and 8 threads a particle, on both sides of the sizes
where the next takes over, against one thread a particle: the same neighbour counts, density
within summation order."""
import numpy as np
import pytest

from paper_2403_11156_gb300 import scenes, sph

from gpu_util import gpu_ctx

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [9728, 9729, 19_456, 19_457, 25_003, 38_912])
def test_groups_equal_one_thread(n):
    out = []
    for lanes in (8, 1):
        d = dict(scenes.dam_break_small(seed=4, n=(35, 34, 33), box=0.8), lanes_per_particle=lanes)
        x = np.array(d["fluid_x"], np.float32)
        d["fluid_x"] = x[np.random.default_rng(n).permutation(len(x))[:n]]
        d.update(divergence_solve=0, warm_start=scenes.WARM_ZERO, min_iter_density=0, max_iter_density=0)
        g = gpu_ctx(d)
        g.sph_steps(1, 1e-6)
        g.sph_synchronize(raise_on_error=False)
        st = g.sph_get_stats(0)
        out.append((g.sph_read_field(sph.FIELD_NN_FLUID), g.sph_read_field(sph.FIELD_NN_BOUNDARY),
                    g.sph_read_field(sph.FIELD_RHO), st["max_fluid_nbrs"], st["max_boundary_nbrs"], st["flags"]))
    a, b = out
    np.testing.assert_array_equal(a[0], b[0])
    np.testing.assert_array_equal(a[1], b[1])
    # FP32 sums of at most 160 positive terms in two orders
    np.testing.assert_allclose(a[2], b[2], rtol=1e-5)
    assert a[3:] == b[3:]
