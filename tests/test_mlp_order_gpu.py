"""The network's sums keep their order: ascending, in one FP32 accumulator.  A training
step shows it (Adam's first steps divide a gradient by its own magnitude, so a bias whose
gradient cancels over the batch turns the last bits of the sum into a visible step).

Reference: the same sums in NumPy.  A fused multiply-add is the FP32 rounding of the exact
product (FP64 holds it) plus the accumulator, whose own FP64 rounding changes the result in
one of some 2^29 cases; sums and products must agree in every bit.
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
gbg = pytest.importorskip("paper_1603_09616_gb300")
from paper_1603_09616_gb300 import surrogate as sg  # noqa: E402


def fma_sum(x, y, start=0.0):
    """sum_k x[k] y[k] over the leading axis, broadcast over the others."""
    acc = np.float32(start)
    for a, b in zip(x.astype(np.float64), y.astype(np.float64)):
        acc = (a * b + acc).astype(np.float32)
    return acc


@pytest.mark.parametrize("dims,batch", [((64, 128, 128, 128, 2), 2048), ((64, 128, 128, 128, 2), 65),
                                        ((5, 7, 33, 128, 3), 301), ((128, 128, 120, 24, 128), 17)])
def test_sums_in_order(dims, batch):
    net = sg.MLP(dims=dims, seed=3)
    rng = np.random.default_rng(batch)
    x = rng.normal(size=(batch, dims[0])).astype(np.float32)
    dy = rng.normal(size=(batch, dims[-1])).astype(np.float32)
    dy -= dy.mean(0)  # the bias gradients cancel over the batch
    xt, dyt = torch.as_tensor(x).cuda(), torch.as_tensor(dy).cuda()
    net.b[0].copy_(torch.as_tensor(rng.normal(size=dims[1]).astype(np.float32)))
    y = net.forward(xt).cpu().numpy()
    net.backward(xt, dyt)
    ws, at, P, A, G = net._workspace(batch).cpu().numpy(), 0, [], [], []
    for n in dims[1:]:  # per layer: pre-activation, activation, gradient
        for kind in (P, A, G):
            kind.append(ws[at:at + batch * n].reshape(batch, n))
            at += batch * n
    w = [t.to(torch.bfloat16).float().cpu().numpy() for t in net.w]
    b = [t.cpu().numpy() for t in net.b]
    G[-1], A[-1] = dy, y
    for l in range(4):
        inp = x if l == 0 else A[l - 1]
        assert np.array_equal(P[l], fma_sum(inp.T[:, :, None], w[l].T[:, None, :]) + b[l])
        assert np.array_equal(net.gb[l].cpu().numpy(), np.add.accumulate(G[l], axis=0)[-1])
        assert np.array_equal(net.gw[l].cpu().numpy(), fma_sum(G[l][:, :, None], inp[:, None, :]))
    # gradients of the activations: G_{l-1} over the activation's slope, which is below 1.13
    # and one rounding away
    for l in range(1, 4):
        dx = fma_sum(G[l].T[:, :, None], w[l][:, None, :]).astype(np.float64)
        p = torch.as_tensor(P[l - 1]).double().requires_grad_()
        torch.nn.functional.gelu(p).sum().backward()
        assert (np.abs(G[l - 1] - dx * p.grad.numpy()) <= 1e-6 * np.abs(dx)).all()
