"""The training loss of the FP16 mode at the ends of its weights' and differences' range: FP64 per element or as good
as that. With parameters of zero the prediction is the input, so that the loss is mean(w (x - target)^2) of
FP32 values; its FP64 sum in any order is within 1e-13 (a few times 2^-53 per addition of a tree).
"""
import numpy as np
import pytest

from paper_2407_12263_gb300 import build as cuda_build
from paper_2407_12263_gb300 import lbm

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


# products of 1e-36, whose rounding errors are below FP32's normal numbers; ordinary ones; and 160^3 products of
# 8e35, of which a thread sums more than FP32 holds
@pytest.mark.parametrize("n,scale,weight", [(16, 1e-12, 1.1e-12), (16, 1e-11, 1e-11), (16, 1e-9, 1e-9), (24, 1.0, 1.0), (16, 3e-10, 1e5),
                                            (16, 1e9, 1e9), (160, 8.3e11, 9.9e11)])
def test_loss_at_the_ends_of_its_range(n, scale, weight):
    cuda_build.build()
    s = torch.cuda.Stream()
    torch.manual_seed(7)
    with torch.cuda.stream(s):
        x = torch.zeros((1, 5, n, n, n), device="cuda")
        target = (torch.rand((1, 5, n, n, n), device="cuda") * 0.2 + 1.0) * scale
        target *= torch.where(torch.rand_like(target) < 0.5, -1.0, 1.0)
        net = lbm.Net(fp16=True, seed=1, stream=s.cuda_stream)
        net.set_params(np.zeros(net.param_count, dtype=np.float32))
        w = np.float32(weight) * np.array([1.0, 1.0, 1.0, 1.0, 1.0] if n == 160 else [1.0, 0.5, 0.0, 1.0, 0.25], dtype=np.float32)
        net.set_loss_weights(w)
        loss = net.gradients(x.data_ptr(), target.data_ptr(), 1, (n, n, n))
        d2 = (x.double() - target.double()) ** 2
        want = float((d2 * torch.tensor(w.astype(np.float64), device="cuda").view(1, 5, 1, 1, 1)).mean())
    assert loss == pytest.approx(want, rel=1e-13, abs=0.0)
