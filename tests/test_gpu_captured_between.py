"""A caller's captured graph stays valid over the calls that lbm.h lets stand between two replays: direct
steps and the handle's own graphs in even numbers, one odd number and another, an accepted surrogate jump. And
with the caller's own buffers (lbm_create_ext), or in a batch, the state is where the parity of the steps
says, without any capture of the handle.
"""
import numpy as np
import pytest

from paper_2407_12263_gb300 import build as cuda_build
from paper_2407_12263_gb300 import inputs as I
from paper_2407_12263_gb300 import lbm

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

D2, D3 = (64, 64, 1), (32, 24, 20)


@pytest.fixture(scope="module", autouse=True)
def _built():
    cuda_build.build()
    lbm.load()


def _init(g):
    g.init_phi(I.multi_droplet_phi(g.grid, 3, 2, (3.0, 5.0), 4.0), I.smooth_velocity(g.grid, 4, 0.03))


# single steps where the region rule takes none (300 x 290), else several steps per launch
@pytest.mark.parametrize("grid,scheme,steps", [(D2, 0, 10), (D2, 0, 0), ((128, 128, 1), 0, 4), ((40, 37, 1), 0, 32), ((300, 290, 1), 0, 2),
                                               (D2, 1, 10), ((128, 128, 1), 1, 2), (D3, 0, 10), (D3, 0, 0)])
def test_replays_between_direct_calls(grid, scheme, steps):
    f = 2 if grid[2] > 1 else 1
    s = torch.cuda.Stream()
    q = 9 if grid[2] == 1 else 19
    net = lbm.Net(fp16=True, seed=1, stream=s.cuda_stream)
    net.set_params(np.zeros(net.param_count, dtype=np.float32))
    results = []
    for captured in (False, True):
        out = torch.zeros((5,) + tuple(n // f for n in grid[::-1]), device="cuda")
        seen = []
        with lbm.Lattice(grid, q, scheme=scheme, stream=s.cuda_stream) as g:
            _init(g)
            g.step(32)  # the handle's own graph, before anything is captured
            g.step(3)

            def calls():
                g.step(steps)
                if scheme == 0:
                    lbm.lbm_coarse_fields(g.h, f, out.data_ptr())

            def once():
                with torch.cuda.stream(s):
                    if captured:
                        graph.replay()
                    else:
                        calls()
                torch.cuda.synchronize()
                seen.append(out.cpu().numpy().copy())

            if captured:
                torch.cuda.synchronize()
                graph = torch.cuda.CUDAGraph()
                with torch.cuda.graph(graph, stream=s):
                    calls()
            once()
            for between in (4, 2, 32, 50, 64, 12, (3, 5), (1, 31), (33, 1), 14):
                for n in between if isinstance(between, tuple) else (between,):
                    g.step(n)
                once()
            g.graph_prepare()
            if grid[2] > 1:
                for judge_steps in (4, 3):
                    rep = lbm.lbm_surrogate_jump(g.h, net, f, (0.0,) * 5 + (1.0,) * 5, 50, judge_steps, 1.0, 1e9, 1e9)
                    assert rep["accepted"]
                    once()
                assert not lbm.lbm_surrogate_jump(g.h, net, f, (0.0,) * 5 + (1.0,) * 5, 6, 4, 1.0, 1e-30, 1e9)["accepted"]
                once()
            g.step(96)
            once()
            results.append((seen, g.get_pops()))
    for a, b in zip(results[0][0], results[1][0]):
        np.testing.assert_array_equal(a, b)
    for a, b in zip(results[0][1], results[1][1]):
        np.testing.assert_array_equal(a, b)


@pytest.mark.parametrize("n", [2, 12, 32, 64, 5])
def test_callers_buffers_hold_the_state_by_parity(n):
    nbytes = lbm.lbm_state_bytes(9, D2, lbm.LBM_STORAGE_FP32)
    states = []
    for single in (True, False):
        fg = [torch.zeros(nbytes, dtype=torch.uint8, device="cuda") for _ in range(2)]
        torch.cuda.synchronize()
        with lbm.Lattice(D2, 9, buffers=(fg[0].data_ptr(), fg[1].data_ptr(), nbytes)) as g:
            _init(g)
            for k in [1] * n if single else [n]:
                g.step(k)
            g.mass()
            states.append(fg[n % 2].cpu().numpy().copy())
    np.testing.assert_array_equal(*states)


def test_batch_replays_between_steps_of_a_case():
    s = torch.cuda.Stream()
    pops = []
    for captured in (False, True):
        with lbm.Batch([lbm.make_case(D2, 9, 0.8, 0.8, 0.02, 4.0, 1e-3) for _ in range(2)], stream=s.cuda_stream) as b:
            for k in range(2):
                _init(b.case(k))
            b.step(4)
            if captured:
                torch.cuda.synchronize()
                graph = torch.cuda.CUDAGraph()
                with torch.cuda.graph(graph, stream=s):
                    b.step(2)
            for n in (32, 4, 12):
                with torch.cuda.stream(s):
                    graph.replay() if captured else b.step(2)
                torch.cuda.synchronize()
                b.case(0).step(n)
                torch.cuda.synchronize()
            pops.append([a for k in range(2) for a in b.case(k).get_pops()])
    for a, b in zip(*pops):
        np.testing.assert_array_equal(a, b)
