"""Mass and diagnostics on grids of more cells than one wave of their blocks has threads (they stride),
with a ragged end, with and without walls: the sum of phi is exact, the sum of rho phi agrees with FP64
sums of lbm_moments' phi (N terms of one sign: relative error below 2 N 2^-53), the counts of
the spheres are exact, and a non-finite population in the first or last cell is seen.
"""
import numpy as np
import pytest

from oracle import diagnostics as DG
from paper_2407_12263_gb300 import build as cuda_build
from paper_2407_12263_gb300 import inputs as I
from paper_2407_12263_gb300 import lbm

pytestmark = pytest.mark.gpu

GRID = (66, 63, 61)


@pytest.fixture(scope="module", autouse=True)
def _built():
    cuda_build.build()
    lbm.load()


@pytest.mark.parametrize("walls", [0, 5])
@pytest.mark.parametrize("storage", [lbm.LBM_STORAGE_FP32, lbm.LBM_STORAGE_FP16, lbm.LBM_STORAGE_BF16])
def test_mass_and_diagnostics_over_more_than_a_wave(storage, walls):
    with lbm.Lattice(GRID, lbm.LBM_D3Q19, 0.8, 0.8, 0.02, 3.0, 2e-3, 3.0, 1.5, storage=storage, walls=walls) as g:
        g.init_phi(I.multi_droplet_phi(GRID, 3, 4, (5.0, 12.0), 4.0), I.smooth_velocity(GRID, 4, 0.03))
        g.step(3)
        phi, p, u = g.moments()
        sum_phi, sum_rho_phi = g.mass()
        fixed = np.rint(phi * 2.0**30).astype(np.int64)
        assert sum_phi == float(fixed.sum()) / 2.0**30
        want = float(((1.0 + 2.0 * phi) * phi).sum())
        assert sum_rho_phi == pytest.approx(want, rel=2 * phi.size * 2.0**-53 * 2)
        d = g.diagnostics((30.0, 31.0, 32.0), 10.0, 20.0)
        h = DG.diagnostics(phi, p, u, 3.0, (30.0, 31.0, 32.0), 10.0, 20.0, walls)
        assert d["n_in"] == h["n_in"] and d["n_out"] == h["n_out"]
        assert d["max_speed"] == pytest.approx(h["max_speed"], rel=2e-7)
        f, gg = g.get_pops()
        for cell in ((0, 0, 0), tuple(n - 1 for n in GRID[::-1])):
            bad = f.copy()
            bad[(7,) + cell] = np.inf
            g.set_pops(bad, gg)
            with pytest.raises(lbm.LBMError) as e:
                g.mass()
            assert e.value.status == lbm.LBM_ENONFINITE
        g.set_pops(f, gg)
        assert g.mass()[0] == pytest.approx(sum_phi, rel=1e-6)
