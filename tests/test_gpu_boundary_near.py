"""The flags of the cells near a boundary, marked from the boundary's side: bodies that move through
a domain several times larger, with both cell sizes and two scenes, give the fields of the tight
domain bit for bit (the cells' order is the same), and the oracle's boundary neighbour counts."""
import numpy as np
import pytest

import oracle
from paper_2403_11156_gb300 import scenes, sph

from gpu_util import gpu_ctx

pytestmark = pytest.mark.gpu

FIELDS = (sph.FIELD_NN_FLUID, sph.FIELD_NN_BOUNDARY, sph.FIELD_RHO, sph.FIELD_PSI, sph.FIELD_SORTED_ID)


@pytest.mark.parametrize("cell", [0.0, 0.0101])
@pytest.mark.parametrize("lanes", [1, 8])
def test_large_domain_equals_tight_one(cell, lanes):
    def descs(f):
        d = [scenes.dam_break_rigid(seed=3, n=(9, 8, 7), n_boxes=2), scenes.dam_break_small(seed=5, n=(7, 6, 5), box=0.4)]
        return [dict(q, domain_max=[f * v for v in q["domain_max"]], cell_size=cell * (q["radius"] / 0.005),
                     lanes_per_particle=lanes) for q in d]
    tight, large = gpu_ctx(descs(1.0)), gpu_ctx(descs(3.0))
    for _ in range(3):
        for g in (tight, large):
            g.sph_steps(1, 4e-4)
            g.sph_synchronize(raise_on_error=False)
        for k in (0, 1):
            for f in FIELDS:
                np.testing.assert_array_equal(tight.sph_read_field(f, scene=k), large.sph_read_field(f, scene=k))
            for a, b in zip(tight.sph_read_state(k), large.sph_read_state(k)):
                np.testing.assert_array_equal(a, b)
        np.testing.assert_array_equal(tight.sph_read_bodies(0), large.sph_read_bodies(0))
    first = gpu_ctx(descs(3.0))
    first.sph_steps(1, 4e-4)
    for k, d in enumerate(descs(1.0)):
        o = oracle.Scene(d)
        o.step(4e-4)
        np.testing.assert_array_equal(first.sph_read_field(sph.FIELD_NN_BOUNDARY, scene=k), o.get(oracle.NN_B).astype(np.int32))
