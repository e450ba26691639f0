"""The 2D displacement kernel where the lattice pitch changes: the last grids of a compiled pitch, and those past all of them
(228 and 229: a run-time pitch with 12 stacked targets; 230 to 233: 8), against the tile-pair kernel, with stored weights
bit for bit.  Tolerances as in test_gpu_disp_tiles.py."""
import numpy as np
import pytest

import vie_synth as V

torch = pytest.importorskip("torch")
import paper_1610_00835_gb300 as P  # noqa: E402
from gpu_util import dev, host, rel_l2  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [193, 194, 227, 228, 229, 230])
def test_applies_at_the_edges_of_the_pitches(n):
    m = V.heterogeneous_2d(n=n, seed=33)
    g = dev(np.random.default_rng(n).random(m.N) + 0.5)

    def apply(h):
        y = torch.empty(m.N, dtype=torch.float64, device="cuda:0")
        P.vie_apply(h, P.VIE_OP_K_SIGMA_S, g, y)
        return host(y)

    h = P.vie_create(2, n, m.sigma_t, m.sigma_s)
    assert P.vie_get_kernel(h) == P.VIE_KERNEL_DISPLACEMENT
    got = apply(h)
    ref = apply(P.vie_create(2, n, m.sigma_t, m.sigma_s, kernel=P.VIE_KERNEL_SYMMETRIC))
    assert rel_l2(got, ref) < 2e-5
    assert np.max(np.abs(got - ref)) < 1e-4 * np.max(np.abs(ref))
    P.vie_assemble(h, P.VIE_OPERATOR_PAIRS32)
    np.testing.assert_array_equal(apply(h), got)
