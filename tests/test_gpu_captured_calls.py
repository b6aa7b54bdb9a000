"""Calls captured into a CUDA graph by their caller give, replayed, the bits of the calls made directly. Kernels
launched one into the next follow a copy, a fill, nothing, or another stream's work there, and an
even number of steps ends in the buffer it began in, whatever the number of its launches, so that
the graph can be replayed again.
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


@pytest.mark.parametrize("n", [2, 8, 10, 32])
@pytest.mark.parametrize("grid,scheme", [((64, 64, 1), 0), ((64, 48, 1), 1), ((150, 140, 1), 0), ((300, 290, 1), 0), ((33, 20, 12), 0),
                                         ((20, 14, 12), 1)])
def test_captured_steps_replay(grid, scheme, n):
    s = torch.cuda.Stream()
    pops = []
    for captured in (False, True):
        with lbm.Lattice(grid, 9 if grid[2] == 1 else 19, scheme=scheme, stream=s.cuda_stream) as g:
            g.init_phi(I.multi_droplet_phi(grid, 3, 2, (3.0, 5.0), 4.0), I.smooth_velocity(grid, 4, 0.03))
            g.step(3)
            if captured:
                torch.cuda.synchronize()
                graph = torch.cuda.CUDAGraph()
                with torch.cuda.graph(graph, stream=s):
                    g.step(n)
                with torch.cuda.stream(s):
                    for _ in range(3):
                        graph.replay()
                torch.cuda.synchronize()
            else:
                g.step(3 * n)
            pops.append(g.get_pops())
    for a, b in zip(*pops):
        np.testing.assert_array_equal(a, b)


def test_captured_surrogate_calls_replay():
    grid, f = (32, 24, 20), 2
    grid_c = tuple(n // f for n in grid)
    s, other = torch.cuda.Stream(), torch.cuda.Stream()
    torch.manual_seed(5)
    x0 = torch.randn((1, 5) + grid_c[::-1], device="cuda")
    x, y, c, done = torch.empty_like(x0), torch.empty_like(x0), torch.empty_like(x0), torch.empty_like(x0)
    work = torch.empty(lbm.lbm_project_workspace_bytes(grid_c), dtype=torch.uint8, device="cuda")
    net = lbm.Net(fp16=True, seed=1, stream=s.cuda_stream)
    with lbm.Lattice(grid, 19, storage=lbm.LBM_STORAGE_FP16, stream=s.cuda_stream) as g:
        g.init_phi(I.droplet_phi(grid, 6.0, 4.0), I.smooth_velocity(grid, 4, 0.03))

        def calls():
            x.copy_(x0)                                     # a copy before the first kernel
            net.forward(x.data_ptr(), y.data_ptr(), 1, grid_c)
            ready = torch.cuda.Event()
            ready.record(s)
            other.wait_event(ready)
            with torch.cuda.stream(other):                  # another stream's work before the next
                done.copy_(y * 0.01)
                joined = torch.cuda.Event()
                joined.record(other)
            s.wait_event(joined)
            assert lbm.lbm_project_solenoidal(done[0, 1].data_ptr(), grid_c, work.data_ptr(), work.numel(), s.cuda_stream) == lbm.LBM_OK
            g.step(2)
            lbm.lbm_coarse_fields(g.h, f, c.data_ptr())
            c[0, 1:4] += done[0, 1:4]

        results = []
        f0, g0 = g.get_pops()
        with torch.cuda.stream(s):
            calls()
            calls()
        torch.cuda.synchronize()
        results.append([t.clone() for t in (y, c, done)])
        g.set_pops(f0, g0)
        torch.cuda.synchronize()
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph, stream=s):
            calls()
        with torch.cuda.stream(s):
            graph.replay()
            graph.replay()
        torch.cuda.synchronize()
        for a, b in zip(results[0], (y, c, done)):
            assert torch.equal(a, b)
