"""The sweep on grids that end inside a tile, along axes, on thick cells and in vacuum, against the oracle."""
import numpy as np
import pytest

import oracle as O
import vie_synth as V

torch = pytest.importorskip("torch")
import paper_1610_00835_gb300 as P  # noqa: E402
from gpu_util import dev, host, rel_l2  # noqa: E402

pytestmark = pytest.mark.gpu


# sigma scale: 0 vacuum; 1 the usual media; 60 steps of optical depth above 1/2 beside thin ones
@pytest.mark.parametrize("scale", [0.0, 1.0, 60.0])
@pytest.mark.parametrize("dim,n", [(2, 1), (2, 2), (2, 15), (2, 16), (2, 17), (2, 33), (3, 1), (3, 3), (3, 8), (3, 9),
                                   (3, 13)])
def test_sweep_matches_oracle(dim, n, scale):
    rng = np.random.default_rng([dim, n])
    N = n ** dim
    st = scale * rng.uniform(0.05, 1.0, N)
    ss, U, f = 0.5 * st, rng.uniform(0.0, 1.0, N), rng.uniform(0.0, 1.0, N)
    axes = np.concatenate([np.eye(dim), -np.eye(dim)])
    dirs = np.concatenate([axes, V.directions(dim, 9)]).astype(np.float32)
    h = P.vie_create(dim, n, st, ss)
    Phi = torch.empty(len(dirs) * N, dtype=torch.float32, device="cuda:0")
    P.ert_sweep(h, dev(U), dev(f), torch.as_tensor(dirs, device="cuda:0"), Phi)
    want = O.sweep(dim, st, ss * U + f, dirs.astype(np.float64))
    assert rel_l2(host(Phi).reshape(len(dirs), -1), want) < 1e-5  # the FP32 bar of the sweep
