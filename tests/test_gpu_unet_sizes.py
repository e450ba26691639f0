"""The network's training step at the edges of its tensor-core tiles: levels down
to one pixel, widths that are no multiple of 16, two segments per row, a smaller
batch after a larger one, and 16 channels (only an adjoint on the tensor cores).

Biases of +1 and -1 with small weights keep every pre-activation away from zero
(half of the channels on, half off), so that rounding flips no ReLU mask.  The
bound: the tensor cores' accumulation truncates, up to 216 additions of 2^-24
each per layer, 1.3e-5, over at most 10 layers forward; the input gradients
keep 16 bits, 2^-16 per layer backward: together 2.9e-4 of the FP64 reference,
5e-4 allowed.  A tap or a row of pixels left out changes a gradient by 1e-2."""
import numpy as np
import pytest

from oracle import unet as R

torch = pytest.importorskip("torch")
import paper_1610_00835_gb300 as P  # noqa: E402
from gpu_util import dev, host, rel_l2  # noqa: E402

pytestmark = pytest.mark.gpu
TOL = 5e-4


def make_params(rng, levels, channels):
    out = []
    for co, ci, k in R.layer_shapes(levels, channels):
        head = k == 1
        out.append((0.3 if head else 0.01) * rng.standard_normal((co, ci, k, k)).astype(np.float32))
        out.append(np.full(co, 0.1, np.float32) if head else np.where(np.arange(co) % 2 == 0, 1, -1).astype(np.float32))
    return out


@pytest.mark.parametrize("levels,channels,n,batches", [(1, 32, 8, (3,)), (1, 32, 1, (1,)), (2, 32, 2, (1,)),
                                                       (4, 32, 8, (3, 1)), (3, 32, 20, (3, 2)), (2, 32, 72, (2,)),
                                                       (3, 32, 136, (2, 1)), (2, 16, 16, (2,))])
def test_gradients_match_reference(levels, channels, n, batches):
    rng = np.random.default_rng(100 * levels + n)
    u = P.vie_unet_create(levels, channels, seed=5)
    pr = make_params(rng, levels, channels)
    P.vie_unet_set_params(u, np.concatenate([q.ravel() for q in pr]))
    pr = [q.astype(np.float64) for q in pr]
    for B in batches:
        x = rng.random((B, 3, n, n)).astype(np.float32)
        t = rng.standard_normal((B, 1, n, n)).astype(np.float32)
        loss_ref, grads_ref, o_ref = R.loss_and_grads(pr, x.astype(np.float64), t.astype(np.float64), levels)
        xd, td = dev(x.ravel(), torch.float32), dev(t.ravel(), torch.float32)
        loss, g = P.vie_unet_loss_grad(u, xd, td, B, n)
        assert loss == pytest.approx(loss_ref, rel=TOL)
        off = 0
        for i, gr in enumerate(grads_ref):
            assert rel_l2(g[off:off + gr.size], gr.ravel()) < TOL, (B, i)
            off += gr.size
        # the BF16 inference hands over the same way: 8 bits per value
        o = torch.empty(B * n * n, dtype=torch.float32, device="cuda:0")
        P.vie_unet_forward(u, xd, o, B, n, use_bf16=True)
        assert rel_l2(host(o), o_ref.ravel()) < 2e-2
