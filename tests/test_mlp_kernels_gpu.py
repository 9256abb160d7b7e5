"""The network's kernels at the sizes where their tiles can go wrong: batches around
the 16-sample blocks and the 128-sample slices, widths that fill no fragment.

Reference: autograd in FP64 on the same BF16 weights.  Tolerance 1e-4 of an array's
largest entry: a worst-case 128 roundings of 2^-24 per product row are 8e-6, times
the four layers and the ratio of a row's absolute sum to its value (< 3 for these
inputs).
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
gbg = pytest.importorskip("paper_1603_09616_gb300")
from paper_1603_09616_gb300 import surrogate as sg  # noqa: E402


@pytest.mark.parametrize("dims", [(64, 128, 128, 128, 2), (5, 7, 33, 128, 3), (1, 16, 17, 64, 1), (128, 120, 24, 8, 128)])
@pytest.mark.parametrize("batch", [1, 16, 129, 545])
def test_network_matches_autograd(dims, batch):
    net = sg.MLP(dims=dims, seed=2)
    rng = np.random.default_rng(batch)
    for b in net.b:
        b.copy_(torch.as_tensor(rng.normal(0, 0.2, b.shape).astype(np.float32)))
    x = torch.as_tensor(rng.normal(size=(batch, dims[0])).astype(np.float32)).cuda()
    dy = torch.as_tensor(rng.normal(size=(batch, dims[-1])).astype(np.float32)).cuda()
    y = net.forward(x)
    net.backward(x, dy)
    w = [t.to(torch.bfloat16).double().requires_grad_() for t in net.w]
    b = [t.double().requires_grad_() for t in net.b]
    a = x.double()
    for l in range(4):
        a = a @ w[l].T + b[l]
        if l < 3:
            a = torch.nn.functional.gelu(a)
    a.backward(dy.double())
    for got, want in [(y, a.detach())] + [(net.gw[l], w[l].grad) for l in range(4)] + [(net.gb[l], b[l].grad) for l in range(4)]:
        assert (got.double() - want).abs().max() <= 1e-4 * want.abs().max()
