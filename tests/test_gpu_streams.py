"""What a call prepares is there for the next call whatever stream that one takes."""
import numpy as np
import pytest

import vie_synth as V

torch = pytest.importorskip("torch")
import paper_1610_00835_gb300 as P  # noqa: E402
from gpu_util import dev, host  # noqa: E402

pytestmark = pytest.mark.gpu


# 25 cells a side: the coarsest grid is the only one, its matrix the largest kept; 200 = 8 x 25
@pytest.mark.parametrize("n", [25, 200])
def test_diffusion_preconditioner_set_on_one_stream_applied_on_another(n):
    v = dev(np.random.default_rng(n).standard_normal(n * n))
    set_on, apply_on = torch.cuda.Stream(), torch.cuda.Stream()
    for seed in range(4):
        # (the buffers come from the medium before, with its matrix in them)
        m = V.bump_medium(2, n, 4, 0.9, seed=5600 + seed)
        h = P.vie_create(2, n, m.sigma_t, m.sigma_s)
        z, want = torch.empty_like(v), torch.empty_like(v)
        torch.cuda.synchronize()
        P.vie_set_diffusion_preconditioner(h, stream=set_on)
        P.vie_diffusion_precondition(h, v, z, stream=apply_on)
        torch.cuda.synchronize()
        P.vie_diffusion_precondition(h, v, want, stream=set_on)
        np.testing.assert_array_equal(host(z), host(want))
        P.vie_destroy(h)
