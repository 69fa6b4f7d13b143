"""A scene that has blown up: particles with NaN or infinite coordinates add nothing to the
volume-fraction field, in the tiled kernel and in the general one."""
import numpy as np
import pytest

from paper_2403_11156_gb300 import scenes

from gpu_util import gpu_ctx

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("axes", [(0,), (1,), (2,), (0, 1), (1, 2), (0, 1, 2)])
@pytest.mark.parametrize("value", [float("nan"), float("inf"), float("-inf")])
def test_field_ignores_non_finite_particles(value, axes):
    d = scenes.dam_break_small(seed=9, n=(9, 11, 13), box=0.4)
    x = np.array(d["fluid_x"], np.float32)
    rng = np.random.default_rng(3)
    bad = rng.permutation(len(x))[:60]
    gone, broken = x.copy(), x.copy()
    gone[bad] = 1e6              # far outside: no node within reach
    for a in axes:
        broken[bad, a] = value
    g = gpu_ctx(d)
    h = 4.0 * d["radius"]
    for spacing in (0.25 * h, 0.8 * h):   # the tiled kernel's range, the general one's
        dims = [int(0.44 / spacing) + 1] * 3
        fields = []
        for state in (gone, broken):
            g.sph_write_state(0, x=state)
            fields.append(g.sph_surface_field((-0.02, -0.02, -0.02), spacing, dims).cpu().numpy())
        assert fields[0].max() > 0.5
        np.testing.assert_array_equal(fields[1], fields[0])
