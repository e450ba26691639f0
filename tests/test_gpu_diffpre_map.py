"""The diffusion preconditioner on every kind of coarsest grid that is kept as a matrix (up to 8 a side, odd ones up to 25),
alone and below finer levels, against the oracle: the bound of test_gpu_diffpre.py."""
import numpy as np
import pytest

import vie_synth as V
from oracle import diffusion as Dm

torch = pytest.importorskip("torch")
import paper_1610_00835_gb300 as P  # noqa: E402
from gpu_util import dev, host, rel_l2  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [2, 3, 4, 6, 7, 9, 11, 12, 14, 22, 23, 25, 36, 50])
def test_coarsest_grids(n):
    m = V.bump_medium(2, n, 4, 0.9, seed=5900 + n)
    h = P.vie_create(2, n, m.sigma_t, m.sigma_s)
    P.vie_set_diffusion_preconditioner(h)
    v = np.random.default_rng(n).standard_normal(m.N)
    z = torch.empty(m.N, dtype=torch.float64, device="cuda:0")
    P.vie_diffusion_precondition(h, dev(v), z)
    assert rel_l2(host(z), Dm.precondition(v, m.sigma_t, m.sigma_s, n)) < 1e-12
