"""The tensor-core layers of the surrogate on grids at the edges of their tiles (8 x 16 voxels of a
plane, runs of planes per CTA): extents below a tile, remainders in x and y, one plane, runs that
cross tiles and samples.

A periodic grid repeated k times along an axis is the same network input seen k times: every
output is the same sum in the same order, so the prediction on the repeated grid equals the
repeated prediction bit for bit. The mean loss and its gradients are the same numbers, apart from
FP32 summation and the FP16 rounding of the gradients between layers, whose scale (a power of two
near the number of elements) differs: 2^-11 relative at each of four layers, so 4e-3 of the
largest gradient of an array covers it, and 1e-5 the loss.
"""
import numpy as np
import pytest

from paper_2407_12263_gb300 import build as cuda_build
from paper_2407_12263_gb300 import lbm

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

CHANS = (5, 32, 32, 32, 5)


@pytest.fixture(scope="module", autouse=True)
def _built():
    cuda_build.build()
    lbm.load()


def arrays(flat):
    out, off = [], 0
    for cin, cout in zip(CHANS[:-1], CHANS[1:]):
        for n in (cout * cin * 27, cout):
            out.append(flat[off:off + n])
            off += n
    return out


@pytest.mark.parametrize("grid,times,batch", [((3, 5, 1), (8, 4, 8), 1), ((1, 1, 2), (9, 17, 2), 2), ((9, 17, 2), (2, 2, 5), 3),
                                              ((8, 16, 9), (3, 1, 1), 2), ((31, 7, 21), (1, 3, 2), 1),
                                              ((24, 33, 40), (2, 1, 1), 4)])
def test_repeated_grid_gives_the_repeated_result(grid, times, batch):
    s = torch.cuda.Stream()
    with torch.cuda.stream(s):
        net = lbm.Net(fp16=True, seed=31, stream=s.cuda_stream)
        p = net.get_params()
        p += np.random.default_rng(31).normal(0, 0.01, p.size).astype(np.float32)
        net.set_params(p)
        rng = np.random.default_rng(32)
        x = torch.tensor(rng.normal(0, 1, (batch, 5) + grid[::-1]).astype(np.float32), device="cuda")
        t = x + torch.tensor(rng.normal(0, 0.3, x.shape).astype(np.float32), device="cuda")
        big = tuple(a * b for a, b in zip(grid, times))
        results = []
        for xs, ts, g in ((x, t, grid), (x.repeat(1, 1, *times[::-1]), t.repeat(1, 1, *times[::-1]), big)):
            y = torch.empty_like(xs)
            net.forward(xs.data_ptr(), y.data_ptr(), batch, g)
            loss = net.gradients(xs.data_ptr(), ts.data_ptr(), batch, g)
            results.append((y, loss, arrays(net.get_grads())))
    s.synchronize()
    (y, loss, grads), (yb, loss_b, grads_b) = results
    assert torch.equal(y.repeat(1, 1, *times[::-1]), yb)
    assert loss_b == pytest.approx(loss, rel=1e-5)
    for a, b in zip(grads, grads_b):
        assert np.abs(a - b).max() <= 4e-3 * np.abs(a).max()
