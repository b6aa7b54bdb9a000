"""Coarse fields of grids with more rows than a launch holds blocks in y (65535), which steps and initial fields
take: 65540 coarse rows at a factor that divides 32, and 65540 rows of whole blocks at factor 1. Against
FP64 block means of lbm_moments, with the bound of test_gpu_coarse_fields.
"""
import numpy as np
import pytest

from paper_2407_12263_gb300 import build as cuda_build
from paper_2407_12263_gb300 import lbm

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.fixture(scope="module", autouse=True)
def _built():
    cuda_build.build()
    lbm.load()


@pytest.mark.parametrize("grid,f", [((4, 131080, 4), 2), ((36, 131072, 4), 2), ((130, 65540, 1), 1)])
def test_coarse_fields_of_tall_grids(grid, f):
    with lbm.Lattice(grid, 9 if grid[2] == 1 else 19) as g:
        phi0 = np.zeros(grid[::-1])
        phi0[:, 100:160] = 1.0
        phi0[:, -200:-80] = np.linspace(0.0, 1.0, 120)[None, :, None]
        y = np.arange(grid[1])[None, :, None] * (2 * np.pi / grid[1])
        u0 = np.stack([0.02 * np.sin(7 * y), 0.01 * np.cos(3 * y), 0.0 * y]).repeat(grid[2], 1).repeat(grid[0], 3)
        g.init_phi(phi0, u0)
        g.step(2)
        out = torch.zeros((5,) + tuple(n // f for n in grid[::-1]), device="cuda")
        torch.cuda.synchronize()
        lbm.lbm_coarse_fields(g.h, f, out.data_ptr())
        torch.cuda.synchronize()
        phi, p, u = g.moments()
    fields = np.stack([phi, u[0], u[1], u[2], p])
    nz, ny, nx = out.shape[1:]
    want = fields.reshape(5, nz, f, ny, f, nx, f).mean(axis=(2, 4, 6))
    np.testing.assert_allclose(out.cpu().numpy(), want, rtol=0, atol=2e-7)
