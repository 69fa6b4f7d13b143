"""The one-launch solves of small contexts against the separate kernels that many scenes take:
the same bits, alone and as one of 17 scenes, for every lane count and solver."""
import numpy as np
import pytest

from paper_2403_11156_gb300 import scenes, sph

from gpu_util import gpu_ctx

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("graph", [True, False])
@pytest.mark.parametrize("lanes", [1, 2, 4, 8])
@pytest.mark.parametrize("kw", [dict(warm_start=scenes.WARM_PREVIOUS, min_iter_divergence=3, min_iter_density=5),
                                dict(warm_start=scenes.WARM_ZERO, eta_density=1e-5),
                                dict(warm_start=scenes.WARM_ZERO, pressure_solver=scenes.SOLVER_PCISPH, divergence_solve=0,
                                     min_iter_density=3)])
def test_one_launch_equals_separate_kernels(lanes, kw, graph):
    # 7 x 5 x 3 particles: less than a block; 9 x 11 x 13: several blocks and a ragged one
    sizes = [(7, 5, 3), (9, 11, 13)] + [(3, 3, 2 + k) for k in range(15)]
    descs = [scenes.dam_break_small(seed=2 + k, n=n, box=0.4, lanes_per_particle=lanes, **kw) for k, n in enumerate(sizes)]
    many = gpu_ctx(descs)          # 17 scenes: the separate kernels
    alone = [gpu_ctx(descs[k]) for k in (0, 1)]
    for g in [many] + alone:
        g.sph_set_mode(graph=graph)
        g.sph_steps(4, 4e-4)
        g.sph_synchronize(raise_on_error=False)
    for k, g in enumerate(alone):
        for f in (sph.FIELD_KAPPA, sph.FIELD_KAPPA_V, sph.FIELD_RHO, sph.FIELD_V_DIV):
            np.testing.assert_array_equal(g.sph_read_field(f), many.sph_read_field(f, scene=k))
        np.testing.assert_array_equal(g.sph_read_state(0)[0], many.sph_read_state(k)[0])
        a, b = g.sph_get_stats(0), many.sph_get_stats(k)
        for key in ("div_iters", "dens_iters", "div_err", "dens_err", "dens_err0", "total_dens_iters", "flags"):
            assert a[key] == b[key], key
