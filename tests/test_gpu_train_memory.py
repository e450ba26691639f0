"""A training batch that fits without the kept split inputs is taken without them, with the same loss and gradients."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
import paper_1610_00835_gb300 as P  # noqa: E402
from gpu_util import rel_l2  # noqa: E402

pytestmark = pytest.mark.gpu


def test_training_step_in_little_memory():
    n, B, levels = 128, 64, 4
    x = torch.randn(B * 3 * n * n, dtype=torch.float32, device="cuda:0")
    t = torch.randn(B * n * n, dtype=torch.float32, device="cuda:0")
    o = torch.empty(B * n * n, dtype=torch.float32, device="cuda:0")
    u = P.vie_unet_create(levels, 32, seed=7)
    want, g_want = P.vie_unet_loss_grad(u, x, t, B, n)  # (all kernels loaded)
    P.vie_unet_destroy(u)
    u = P.vie_unet_create(levels, 32, seed=7)
    P.vie_unet_forward(u, x, o, B, n, use_bf16=True)  # the activations are allocated
    P.vie_release_memory()
    torch.cuda.empty_cache()
    torch.cuda.synchronize()
    # the kept inputs of this batch take 1.5 GB, the CUDA-core form's planes 0.5 GB
    free = torch.cuda.mem_get_info()[0]
    hog = torch.empty(free - (900 << 20), dtype=torch.uint8, device="cuda:0")
    try:
        loss, g = P.vie_unet_loss_grad(u, x, t, B, n)
    finally:
        del hog
        torch.cuda.empty_cache()
    assert loss == want  # the same forward, bit for bit
    off = 0
    for i in range(2 * levels + 2 * (levels - 1)):
        co, ci = 32, 3 if i == 0 else 64 if i >= 2 * levels and i % 2 == 0 else 32
        for size in (co * ci * 9, co):
            # the same masks and input gradients; sums in FP32 here, on the tensor cores there (4e-7 of the exact ones each)
            assert rel_l2(g[off:off + size], g_want[off:off + size]) < 2e-6, i
            off += size
    assert off + 33 == g.size
    np.testing.assert_array_equal(g[off:], g_want[off:])
