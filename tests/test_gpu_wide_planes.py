"""16-bit D3Q19 grids around 2^29 cells, where a plane of the state passes 4 GiB and the step leaves 32-bit
offsets for 64-bit ones: the largest grid of the one form and the smallest of the other, each several copies in z
of a smaller periodic grid, whose state they must repeat bit for bit.
"""
import numpy as np
import pytest

from paper_2407_12263_gb300 import build as cuda_build
from paper_2407_12263_gb300 import lbm

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

GENERAL = dict(walls=3, rho_ratio=3.0, mu_ratio=1.5, body_force=(1e-5, -2e-5, 0.0))
NX = NY = 512


def _state(nz, phi0, steps, storage, **kw):
    grid = (NX, NY, nz)
    nbytes = lbm.lbm_state_bytes(19, grid, storage)
    fg = [torch.empty(nbytes, dtype=torch.uint8, device="cuda") for _ in range(2)]
    torch.cuda.synchronize()
    with lbm.Lattice(grid, 19, storage=storage, sigma=0.01, buffers=(fg[0].data_ptr(), fg[1].data_ptr(), nbytes), **kw) as g:
        g.init_phi(phi0)
        g.step(steps)
        torch.cuda.synchronize()
    return fg[steps % 2].view(torch.int64).view(10, nz, NY, NX)  # the moments, then a word of 8 bytes per pair


@pytest.mark.parametrize("nz,copies,storage,kw", [
    (256, 8, lbm.LBM_STORAGE_FP16, {}),
    (256, 8, lbm.LBM_STORAGE_BF16, GENERAL),
    (256, 8, lbm.LBM_STORAGE_FP16, dict(scheme=lbm.LBM_SCHEME_FINITE_DIFFERENCE)),
    (89, 23, lbm.LBM_STORAGE_FP16, GENERAL),
    (89, 23, lbm.LBM_STORAGE_BF16, dict(scheme=lbm.LBM_SCHEME_FINITE_DIFFERENCE))])
def test_steps_of_planes_around_4_gib(nz, copies, storage, kw):
    cuda_build.build()
    z, y, x = (2 * np.pi * np.arange(n) / n for n in (nz, NY, NX))
    # a mean clearly below 1/2: the bulk phase that g is stored relative to follows from it
    phi0 = 0.42 + 0.3 * np.sin(3 * z)[:, None, None] * np.cos(20 * y + 0.3)[:, None] * np.sin(17 * x + np.cos(2 * x)) \
        + 0.1 * np.cos(5 * z + 0.7)[:, None, None]
    small = _state(nz, phi0, 3, storage, **kw)
    big = _state(nz * copies, np.tile(phi0, (copies, 1, 1)), 3, storage, **kw)
    assert (big.numel() // 10 >= 1 << 29) == (copies == 8)
    for k in range(10):
        for c in range(copies):
            assert torch.equal(big[k, c * nz:(c + 1) * nz], small[k]), (k, c)
    del big
    torch.cuda.empty_cache()
