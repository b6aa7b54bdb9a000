"""lbm_launch_count over an accepted jump: the launches of its parts on the handle."""
import numpy as np
import pytest

from paper_2407_12263_gb300 import build as cuda_build
from paper_2407_12263_gb300 import inputs as I
from paper_2407_12263_gb300 import lbm

pytestmark = pytest.mark.gpu


# factor 3 does not divide 32: the judge balances in a launch of its own; walls: no projection
@pytest.mark.parametrize("f,walls", [(2, 0), (3, 0), (2, 3)])
def test_launches_of_an_accepted_jump(f, walls):
    cuda_build.build()
    grid, steps = (36, 24, 24), 5
    net = lbm.Net(fp16=True, seed=1)
    net.set_params(np.zeros(net.param_count, dtype=np.float32))
    with lbm.Lattice(grid, 19, walls=walls) as g:
        g.init_phi(I.droplet_phi(grid, 6.0, 4.0), I.smooth_velocity(grid, 4, 0.03))
        before = g.launch_count
        assert lbm.lbm_surrogate_jump(g.h, net, f, (0.0,) * 5 + (1.0,) * 5, 50, steps, 1.0, 1e9, 1e9)["accepted"]
        sum_phi, coarse, measures, restart, rates = 2, 1, 1, 2, 2
        # twiddles, a pass along each axis, the modes, a pass back along each axis
        project = 0 if walls else 1 + 3 + 1 + 3
        one = restart + (2 if f == 2 else 3) + steps + rates
        assert g.launch_count - before == sum_phi + coarse + project + measures + 2 * one
