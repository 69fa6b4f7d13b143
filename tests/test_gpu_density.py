"""The one-thread density sweep (half-precision candidate filter, exact predicate after) against
the eight-lane sweep (exact predicate only): neighbour counts, their maximum and the overflow
flag equal, density within summation order, where the filter is tight, loose, off or overrun."""
import numpy as np
import pytest

from paper_2403_11156_gb300 import scenes, sph

from gpu_util import gpu_ctx

pytestmark = pytest.mark.gpu


def _scene(shift, cap, crowd, away, lanes, cell):
    d = dict(scenes.dam_break_small(seed=4, n=(13, 11, 12), box=0.4), lanes_per_particle=lanes, max_fluid_neighbors=cap)
    if cell:
        d["cell_size"] = cell
    x = np.array(d["fluid_x"], np.float32)
    rng = np.random.default_rng(1)
    x += rng.uniform(-0.004, 0.004, x.shape).astype(np.float32)
    if crowd:      # 300 particles in one cell: rows of several masks, lists overrun
        x[:300] = x[700] + rng.uniform(-0.004, 0.004, (300, 3)).astype(np.float32)
    if away:       # far outside the domain, in one another's reach
        x[5:25] = (np.float32(away) + rng.uniform(0, 0.02, (20, 3))).astype(np.float32)
    d["fluid_x"] = x + np.float32(shift)
    d["boundary_x"] = np.asarray(d["boundary_x"], np.float32) + np.float32(shift)
    for k in ("domain_min", "domain_max"):
        d[k] = [float(v) + shift for v in d[k]]
    d.update(divergence_solve=0, warm_start=scenes.WARM_ZERO, min_iter_density=0, max_iter_density=0)
    return d


@pytest.mark.parametrize("cell", [0.0, 0.0201])
@pytest.mark.parametrize("shift,cap,crowd,away", [
    (0.0, 0, False, 0.0), (0.0, 12, False, 0.0), (0.0, 1, False, 0.0), (0.0, 0, True, 0.0), (0.0, 0, False, 3.0),
    (0.0, 0, False, 3000.0), (0.0, 0, False, -4e8), (60.0, 0, False, 0.0), (-4000.0, 0, False, 0.0)])
def test_filter_keeps_every_neighbour(shift, cap, crowd, away, cell):
    out = []
    for lanes in (8, 1):
        g = gpu_ctx(_scene(shift, cap, crowd, away, lanes, cell))
        g.sph_steps(1, 1e-6)
        g.sph_synchronize(raise_on_error=False)
        st = g.sph_get_stats(0)
        out.append((g.sph_read_field(sph.FIELD_NN_FLUID), g.sph_read_field(sph.FIELD_NN_BOUNDARY),
                    g.sph_read_field(sph.FIELD_RHO), st["max_fluid_nbrs"], st["max_boundary_nbrs"], st["flags"]))
    a, b = out
    np.testing.assert_array_equal(a[0], b[0])
    np.testing.assert_array_equal(a[1], b[1])
    # FP32 sums of at most 1024 positive terms in two orders
    np.testing.assert_allclose(a[2], b[2], rtol=1e-5)
    assert a[3:] == b[3:]
