"""Several steps of a small D2Q9 grid in one launch give the bits of single steps: lbm_step(n) against
n calls of lbm_step(1), which are always single launches. Grids: the smallest, sides that are no
multiple of a tile, thin ones, and the largest for which each region size is taken; walls on
one or both axes, density and viscosity ratio and gravity; step counts that split unevenly, with
and without graphs.
"""
import numpy as np
import pytest

from paper_2407_12263_gb300 import build as cuda_build
from paper_2407_12263_gb300 import inputs as I
from paper_2407_12263_gb300 import lbm

pytestmark = pytest.mark.gpu

GENERAL = dict(rho_ratio=3.0, mu_ratio=1.5, body_force=(1e-5, -2e-5, 0.0))


@pytest.fixture(scope="module", autouse=True)
def _built():
    cuda_build.build()
    lbm.load()


def _run(grid, calls, **kw):
    with lbm.Lattice(grid, 9, **kw) as g:
        g.init_phi(I.multi_droplet_phi(grid, 3, 2, (3.0, 6.0), 4.0), I.smooth_velocity(grid, 4, 0.03))
        n0 = g.launch_count
        for n in calls:
            g.step(n)
        launches = g.launch_count - n0
        return g.get_pops(), g.mass()[0], launches


@pytest.mark.parametrize("walls,general", [(0, {}), (1, {}), (3, GENERAL), (0, GENERAL)])
@pytest.mark.parametrize("storage", [lbm.LBM_STORAGE_FP32, lbm.LBM_STORAGE_FP16, lbm.LBM_STORAGE_BF16])
@pytest.mark.parametrize("scheme", [lbm.LBM_SCHEME_DIFFERENCE_FREE, lbm.LBM_SCHEME_FINITE_DIFFERENCE])
@pytest.mark.parametrize("grid", [(3, 3, 1), (41, 37, 1), (7, 150, 1), (97, 96, 1), (131, 120, 1), (216, 210, 1),
                                  (280, 250, 1)])
def test_several_steps_per_launch_are_single_steps(grid, scheme, storage, walls, general):
    kw = dict(scheme=scheme, storage=storage, walls=walls, **general)
    (f, g), mass, single = _run(grid, [1] * 46, graph_steps=0, **kw)
    assert single == 46 * (1 + scheme)
    for graph_steps, calls in ((0, (2, 7, 37)), (32, (41, 5)), (2, (46,))):
        (f2, g2), mass2, launches = _run(grid, calls, graph_steps=graph_steps, **kw)
        np.testing.assert_array_equal(f, f2)
        np.testing.assert_array_equal(g, g2)
        assert mass == mass2
        assert launches <= single
        if graph_steps == 0 and max(grid) < 200:
            assert launches < single
