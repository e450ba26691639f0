"""Gradients that are sums over many pixels: equal terms round the same way each time, so a long FP32 chain drifts.

Weights of zero leave constant planes: every term of a bias's or a head weight's gradient is the same number.  64 of them
in FP32 lose at most sum_k k / 64 2^-24 = 1.9e-6 of their sum; the rest is FP64, and the result FP32: 2e-6 allowed."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
import paper_1610_00835_gb300 as P  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,B", [(512, 16), (520, 3)])
def test_bias_and_head_gradients_of_large_images(n, B):
    u = P.vie_unet_create(1, 32, seed=1)
    rng = np.random.default_rng(3)
    w1, w2, head = 32 * 27, 32 * 288, 32
    p = np.zeros(w1 + 32 + w2 + 32 + head + 1, np.float32)
    b2 = w1 + 32 + w2
    e = rng.uniform(0.5, 2.0, 32).astype(np.float32)
    wh = rng.uniform(0.01, 0.1, 32).astype(np.float32)
    p[b2:b2 + 32], p[b2 + 32:b2 + 64], p[-1] = e, wh, 0.1
    P.vie_unet_set_params(u, p)
    x = torch.rand(B * 3 * n * n, dtype=torch.float32, device="cuda:0")
    t = torch.zeros(B * n * n, dtype=torch.float32, device="cuda:0")
    _, g = P.vie_unet_loss_grad(u, x, t, B, n)
    o = torch.empty(B, 1, n, n, device="cuda:0")
    P.vie_unet_layer_io(u, 2, None, o)
    go = 2.0 * o / np.float32(B * n * n)  # as the loss forms it, in FP32
    assert float(go.min()) == float(go.max())
    total = float(go.double().sum())
    v = float(go[0, 0, 0, 0])
    want = np.concatenate([[float(np.float32(w) * np.float32(v)) * B * n * n for w in wh], total * e.astype(np.float64), [total]])
    np.testing.assert_allclose(g[b2:], want, rtol=2e-6)
