"""A bounded wait that runs out in a training step: the call says so, and no parameter moves."""
import os

import numpy as np
import pytest

torch = pytest.importorskip("torch")
import paper_1610_00835_gb300 as P  # noqa: E402

pytestmark = pytest.mark.gpu


def test_training_timeout_is_reported_and_leaves_the_network_alone(tmp_path):
    n, B = 16, 2
    rng = np.random.default_rng(9)
    x = torch.as_tensor(rng.standard_normal(B * 3 * n * n), dtype=torch.float32, device="cuda:0")
    t = torch.as_tensor(rng.standard_normal(B * n * n), dtype=torch.float32, device="cuda:0")
    nets = [P.vie_unet_create(2, 32, seed=4) for _ in range(2)]
    for u in nets:
        P.vie_unet_train_step(u, x, t, B, n, 1e-3)
    u, v = nets

    def file_of(net):  # parameters, step and both moments
        path = os.path.join(tmp_path, "net.bin")
        P.vie_unet_save(net, path)
        with open(path, "rb") as f:
            return f.read()

    before = file_of(u)
    try:
        P.vie_set_wait_limits(1000.0, 0.0)
        for call in (lambda: P.vie_unet_loss_grad(u, x, t, B, n), lambda: P.vie_unet_train_step(u, x, t, B, n, 1e-3)):
            with pytest.raises(P.VieError) as e:
                call()
            assert e.value.status == P.VIE_ERR_TIMEOUT
    finally:
        P.vie_set_wait_limits(1000.0, -1.0)
    assert file_of(u) == before
    # and the next step is the one that a network without the failure takes
    assert P.vie_unet_train_step(u, x, t, B, n, 1e-3) == P.vie_unet_train_step(v, x, t, B, n, 1e-3)
    np.testing.assert_array_equal(P.vie_unet_get_params(u), P.vie_unet_get_params(v))
