"""The weight and bias gradients of one 32-channel layer alone against 64 bits, from the layer's own FP32 input and output
gradient: no worse than FP32 multiply-adds (1.2e-7 to 2.1e-7 relative at these sizes; the six products of the split operands
in one truncating accumulator have 2.0e-7 to 3.7e-7).

A row's large products take 8 truncating additions in a column of their own, each losing 2^-24 of the partial sum on average,
2.7e-7 of the row's sum where all terms have one sign; here they have both, and the rows' losses average out to a third of
that or less: 1.5e-7 allowed.  The bias: 8 FP32 terms a thread, the rest in trees and FP64: 1e-7."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
import paper_1610_00835_gb300 as P  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,B", [(64, 4), (128, 4), (136, 2)])
def test_layer_gradients_keep_fp32_accuracy(n, B):
    u = P.vie_unet_create(1, 32, seed=n)
    rng = np.random.default_rng(n)
    x = torch.as_tensor(rng.standard_normal(B * 3 * n * n), dtype=torch.float32, device="cuda:0")
    t = torch.as_tensor(rng.standard_normal((B, n, n)), dtype=torch.float32, device="cuda:0")
    _, grads = P.vie_unet_loss_grad(u, x, t.reshape(-1), B, n)
    grads = torch.as_tensor(grads, device="cuda:0").double()
    a, e, o = (torch.empty(B, c, n, n, device="cuda:0") for c in (32, 32, 1))
    for layer, out in enumerate((a, e, o)):
        P.vie_unet_layer_io(u, layer, None, out)
    w2 = 32 * 27 + 32  # the second layer's weights, its bias, the head
    b2 = w2 + 32 * 288
    head = torch.as_tensor(P.vie_unet_get_params(u)[b2 + 32:b2 + 64], device="cuda:0")
    go = 2.0 * (o - t[:, None]) / np.float32(B * n * n)  # as the loss forms it, in FP32
    g = torch.where(e > 0, head[None, :, None, None] * go, torch.zeros((), device="cuda:0")).double()
    pad = torch.nn.functional.pad(a.double(), (1, 1, 1, 1))
    dw = torch.stack([torch.einsum("bopq,bipq->oi", g, pad[:, :, k // 3:k // 3 + n, k % 3:k % 3 + n]) for k in range(9)], -1)
    for got, want, tol in ((grads[w2:b2], dw.reshape(-1), 1.5e-7), (grads[b2:b2 + 32], g.sum((0, 2, 3)), 1e-7)):
        assert float((got - want).norm() / want.norm()) < tol
