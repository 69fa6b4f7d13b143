"""The field's grid order works in the context's own sort scratch: the steps after it, the
readable fields and the count and trace of step launches are those without it."""
import numpy as np
import pytest

from paper_2403_11156_gb300 import scenes, sph

from gpu_util import gpu_ctx

pytestmark = pytest.mark.gpu

FIELDS = (sph.FIELD_RHO, sph.FIELD_ALPHA, sph.FIELD_KAPPA, sph.FIELD_NN_FLUID, sph.FIELD_NN_BOUNDARY,
          sph.FIELD_CELL_KEY, sph.FIELD_SORTED_ID, sph.FIELD_KAPPA_PREV, sph.FIELD_PSI)


def _all(g, scene):
    return [g.sph_read_field(f, scene=scene) for f in FIELDS] + list(g.sph_read_state(scene))


@pytest.mark.parametrize("lanes", [1, 2, 8])
def test_steps_around_a_field_are_unchanged(lanes):
    descs = [scenes.dam_break_small(seed=2 + k, n=n, box=0.4, lanes_per_particle=lanes,
                                    warm_start=scenes.WARM_PREVIOUS) for k, n in enumerate([(7, 5, 3), (9, 11, 13)])]
    plain, drawn = gpu_ctx(descs), gpu_ctx(descs)
    for spacing in (0.01, 0.03):
        for g in (plain, drawn):
            g.sph_steps(2, 4e-4)
        for k in (1, 0):
            before = _all(drawn, k)
            drawn.sph_surface_field((0.0, 0.0, 0.0), spacing, (40, 40, 40), scene=k)
            for a, b in zip(_all(drawn, k), before):
                np.testing.assert_array_equal(a, b)
    for g in (plain, drawn):
        g.sph_steps(2, 4e-4)
        g.sph_synchronize(raise_on_error=False)
    for k in (0, 1):
        for a, b in zip(_all(plain, k), _all(drawn, k)):
            np.testing.assert_array_equal(a, b)


def test_field_is_no_step_launch():
    g = gpu_ctx(scenes.dam_break_small(seed=2, n=(9, 11, 13), box=0.4))
    g.sph_steps(1, 4e-4)
    g.sph_set_trace(256)
    n = g.sph_launch_count()
    g.sph_surface_field((0.0, 0.0, 0.0), 0.01, (40, 40, 40))
    assert g.sph_launch_count() == n
    assert g.sph_read_trace(256)[0] == []
