"""A step that the runtime refuses to launch (a block per row of 128 cells, and more rows than a launch holds) leaves
the handle as it was: the state in its buffer, the launch count, and the calls after it.
"""
import numpy as np
import pytest

from paper_2407_12263_gb300 import build as cuda_build
from paper_2407_12263_gb300 import lbm

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("scheme", [lbm.LBM_SCHEME_DIFFERENCE_FREE, lbm.LBM_SCHEME_FINITE_DIFFERENCE])
@pytest.mark.parametrize("graph_steps,n", [(0, 1), (32, 3), (32, 33)])
def test_a_refused_step_changes_nothing(graph_steps, n, scheme):
    cuda_build.build()
    grid = (128, 65600, 1)
    with lbm.Lattice(grid, 9, graph_steps=graph_steps, scheme=scheme) as g:
        phi0 = np.tile(np.linspace(0.0, 1.0, 128), (1, grid[1], 1))
        g.init_phi(phi0)
        launches = g.launch_count
        with pytest.raises(lbm.LBMError) as err:
            g.step(n)
        assert err.value.status == lbm.LBM_ECUDA
        assert g.launch_count == launches
        # the calls after it, the first of them a plain launch, work and see the initial state
        sum_phi = g.mass()[0]
        assert sum_phi == pytest.approx(phi0.sum(), rel=1e-7)
        f, g0 = g.get_pops()
        np.testing.assert_allclose(g0.sum(axis=0)[0], phi0[0], rtol=0, atol=1e-6)
        if scheme == lbm.LBM_SCHEME_DIFFERENCE_FREE:
            out = torch.zeros((5, 1, grid[1], grid[0]), device="cuda")
            torch.cuda.synchronize()
            lbm.lbm_coarse_fields(g.h, 1, out.data_ptr())
            torch.cuda.synchronize()
            assert float(out[0].double().sum()) == pytest.approx(phi0.sum(), rel=1e-6)
