"""lbm_coarse_fields on the GPU for every way it splits the work: factor 1 (one cell per thread),
factors that divide 32 (lanes of a warp), other factors up to 64 (whole coarse cells of a block
row) and larger ones (one coarse cell per thread), on grids that leave partial warps and blocks.

Against FP64 block means of lbm_moments: the output is FP32 (half a unit in the last place of
phi, below 2: 6e-8) and a field of the two kernels may differ in its last FP32 bit (u below
2^-4, p below 1/2: 3e-8; phi is the same integer), so 2e-7 covers both; sums over a block are
kept to well below that (about 48 bits and FP64).
"""
import numpy as np
import pytest

from paper_2407_12263_gb300 import build as cuda_build
from paper_2407_12263_gb300 import inputs as I
from paper_2407_12263_gb300 import lbm

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.fixture(scope="module", autouse=True)
def _built():
    cuda_build.build()
    lbm.load()


@pytest.mark.parametrize("grid,f", [((37, 10, 6), 1), ((131, 5, 4), 1), ((70, 36, 1), 1), ((38, 10, 6), 2),
                                    ((96, 64, 32), 32), ((69, 9, 6), 3), ((195, 10, 5), 5), ((74, 74, 37), 37),
                                    ((65, 65, 65), 65)])
@pytest.mark.parametrize("storage", [lbm.LBM_STORAGE_FP32, lbm.LBM_STORAGE_FP16, lbm.LBM_STORAGE_BF16])
@pytest.mark.parametrize("walls", [0, 3])
def test_coarse_fields_of_every_split(grid, f, storage, walls):
    Q = 9 if grid[2] == 1 else 19
    general = dict(rho_ratio=2.0, mu_ratio=1.5, body_force=(1e-5, -2e-5, 0.0)) if walls else {}
    with lbm.Lattice(grid, Q, storage=storage, walls=walls, **general) as g:
        g.init_phi(I.multi_droplet_phi(grid, 3, 2, (3.0, 5.0), 4.0), I.smooth_velocity(grid, 4, 0.03))
        g.step(3)
        out = torch.empty((5,) + tuple(n // f for n in grid[::-1]), device="cuda")
        torch.cuda.synchronize()
        lbm.lbm_coarse_fields(g.h, f, out.data_ptr())
        torch.cuda.synchronize()
        phi, p, u = g.moments()
    fields = np.stack([phi, u[0], u[1], u[2], p])
    nz, ny, nx = out.shape[1:]
    want = fields.reshape(5, nz, f, ny, f, nx, f).mean(axis=(2, 4, 6))
    np.testing.assert_allclose(out.cpu().numpy(), want, rtol=0, atol=2e-7)
