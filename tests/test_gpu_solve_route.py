"""Which kernels a context's solves run: one launch where all sweep blocks are resident at once,
the separate passes and tests with more scenes or more blocks, seen in the device trace."""
import pytest

from paper_2403_11156_gb300 import scenes

from gpu_util import gpu_ctx

pytestmark = pytest.mark.gpu

ONE = {"div_solve", "dens_solve"}
SEPARATE = {"div_pass_a", "div_pass_b", "div_check", "dens_pass_a", "dens_pass_b", "dens_check"}


@pytest.mark.parametrize("lanes", [1, 2, 4, 8])
@pytest.mark.parametrize("sizes,one", [([(9, 11, 13)], True), ([(5, 4, 3)] * 8, True), ([(5, 4, 3)] * 9, False),
                                       ([(60, 60, 100)], False)])
def test_route(sizes, one, lanes):
    descs = [scenes.dam_break_small(seed=2 + k, n=n, box=2.2, lanes_per_particle=lanes, warm_start=scenes.WARM_ZERO)
             for k, n in enumerate(sizes)]
    g = gpu_ctx(descs)
    g.sph_set_trace(4096)
    g.sph_steps(1, 4e-4)
    g.sph_synchronize(raise_on_error=False)
    names = set(g.sph_read_trace(4096)[0])
    assert (ONE if one else SEPARATE) <= names
    assert not (SEPARATE if one else ONE) & names
