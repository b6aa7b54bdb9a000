"""Steps whose blocks are packed along a plane's cells, whatever its rows, give the bits of blocks of whole
rows. Difference-free: against the same case in a batch, whose tiles are boxes of cells. Finite
difference: a periodic grid of rows of 48 cells (packed) against two copies of it side by side, rows of 96
(not packed). Grids: rows shorter than a warp, one cell more or less than a row or a plane of
blocks, rows of a prime length, and planes of fewer cells than a block.
"""
import numpy as np
import pytest

from paper_2407_12263_gb300 import build as cuda_build
from paper_2407_12263_gb300 import inputs as I
from paper_2407_12263_gb300 import lbm

pytestmark = pytest.mark.gpu

GENERAL = dict(rho_ratio=3.0, mu_ratio=1.5, body_force=(1e-5, -2e-5, 3e-5))
STORAGES = [lbm.LBM_STORAGE_FP32, lbm.LBM_STORAGE_FP16, lbm.LBM_STORAGE_BF16]


@pytest.fixture(scope="module", autouse=True)
def _built():
    cuda_build.build()
    lbm.load()


@pytest.mark.parametrize("storage", STORAGES)
@pytest.mark.parametrize("walls,general", [(0, {}), (4, GENERAL), (7, GENERAL)])
@pytest.mark.parametrize("grid", [(9, 8, 8), (31, 9, 8), (33, 8, 9), (65, 127, 3), (127, 3, 8), (129, 8, 5), (257, 5, 8), (130, 63, 4)])
def test_packed_blocks_against_tiles_of_a_batch(grid, walls, general, storage):
    params = dict(tau_f=0.8, tau_g=0.8, M=0.02, xi=4.0, sigma=1e-3, courant=0.997, walls=walls, storage=storage, **general)
    phi0, u0 = I.multi_droplet_phi(grid, 3, 2, (2.0, 4.0), 4.0), I.smooth_velocity(grid, 4, 0.03)
    batch = lbm.Batch([lbm.make_case(grid, lbm.LBM_D3Q19, **params)], graph_steps=0)
    batch.set_config(0, (8, 8, 2), False)
    batch.case(0).init_phi(phi0, u0)
    batch.step(13)
    with lbm.Lattice(grid, lbm.LBM_D3Q19, graph_steps=0, **params) as g:
        g.init_phi(phi0, u0)
        g.step(13)
        for a, b in zip(batch.case(0).get_pops(), g.get_pops()):
            np.testing.assert_array_equal(a, b)


@pytest.mark.parametrize("storage", STORAGES)
@pytest.mark.parametrize("general", [{}, dict(walls=6, **GENERAL)])
def test_packed_finite_difference_against_two_copies(storage, general):
    grid = (48, 8, 7)
    phi0, u0 = I.multi_droplet_phi(grid, 3, 2, (2.0, 4.0), 4.0), I.smooth_velocity(grid, 4, 0.03)
    pops = []
    for copies in (1, 2):
        n = (grid[0] * copies,) + grid[1:]
        with lbm.Lattice(n, lbm.LBM_D3Q19, scheme=lbm.LBM_SCHEME_FINITE_DIFFERENCE, storage=storage, graph_steps=0, **general) as g:
            g.init_phi(np.concatenate([phi0] * copies, axis=-1), np.concatenate([u0] * copies, axis=-1))
            g.step(13)
            pops.append(g.get_pops())
    for a, b in zip(*pops):
        a, b = np.asarray(a), np.asarray(b)
        b = b.reshape(a.shape[0], *grid[::-1][:2], 2 * grid[0])
        a = a.reshape(a.shape[0], *grid[::-1])
        np.testing.assert_array_equal(b[..., :grid[0]], a)
        np.testing.assert_array_equal(b[..., grid[0]:], a)
