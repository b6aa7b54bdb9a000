"""An accepted jump ends in the state that its own parts build one by one, bit for bit: with a
network of zeros (the prediction is its input) and mean 0, std 1, the prediction is the state's own
coarse fields with the velocity projected, and the state is the restart from it advanced by
judge_steps steps. Even and odd judge_steps end in different buffers; factor 3 does not divide 32
and judges with lbm_coarse_fields instead of lbm_coarse_phi. A second jump starts from the
buffer that the first one ended in.
"""
import numpy as np
import pytest

from paper_2407_12263_gb300 import build as cuda_build
from paper_2407_12263_gb300 import inputs as I
from paper_2407_12263_gb300 import lbm

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

P0 = 1.0 / 3.0


@pytest.fixture(scope="module", autouse=True)
def _built():
    cuda_build.build()
    lbm.load()


def _restart_by_parts(g, f, judge_steps, stream):
    grid_c = tuple(n // f for n in g.grid)
    c = torch.empty((5,) + grid_c[::-1], device="cuda")
    work = torch.empty(lbm.lbm_project_workspace_bytes(grid_c), dtype=torch.uint8, device="cuda")
    torch.cuda.synchronize()
    lbm.lbm_coarse_fields(g.h, f, c.data_ptr())
    assert lbm.lbm_project_solenoidal(c[1].data_ptr(), grid_c, work.data_ptr(), work.numel(), stream) == lbm.LBM_OK
    lbm.lbm_restart_from_coarse(g.h, f, c.data_ptr(), (P0 * 3.0) / 3.0)
    g.step(judge_steps)


@pytest.mark.parametrize("storage", [lbm.LBM_STORAGE_FP32, lbm.LBM_STORAGE_FP16])
@pytest.mark.parametrize("f,judge_steps,grid", [(2, 4, (32, 24, 20)), (2, 3, (36, 16, 28)), (3, 3, (36, 24, 21)),
                                                (3, 8, (24, 27, 30))])
def test_accepted_jump_is_the_sum_of_its_parts(f, judge_steps, grid, storage):
    s = torch.cuda.Stream()
    phi = I.droplet_phi(grid, 6.0, 4.0)
    u = I.smooth_velocity(grid, 4, 0.03)
    with lbm.Lattice(grid, 19, storage=storage, stream=s.cuda_stream) as a, \
            lbm.Lattice(grid, 19, storage=storage, stream=s.cuda_stream) as b:
        for g in (a, b):
            g.init_phi(phi, u, P0)
            g.step(5)
        net = lbm.Net(fp16=True, seed=1, stream=s.cuda_stream)
        net.set_params(np.zeros(net.param_count, dtype=np.float32))
        for _ in range(2):
            rep = lbm.lbm_surrogate_jump(a.h, net, f, (0.0,) * 5 + (1.0,) * 5, 50, judge_steps, 1.0, 1e9, 1e9)
            assert rep["accepted"] and rep["projected"]
            _restart_by_parts(b, f, judge_steps, s.cuda_stream)
            for got, want in zip(a.get_pops(), b.get_pops()):
                np.testing.assert_array_equal(got, want)
            assert a.mass()[0] == b.mass()[0]
        a.step(2)
        b.step(2)
        np.testing.assert_array_equal(a.get_pops()[1], b.get_pops()[1])
