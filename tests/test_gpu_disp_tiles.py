"""The displacement kernels at the edges of their tiles, tile pairs and lattice
pitches: every row against the tile-pair kernel, some against the oracle.

Tolerances: each kernel holds 1e-5 relative L2 against the FP64 oracle, so two
of them differ by at most 2e-5; a pair left out or taken twice is of order
1 / n^2 of a row or more and shows in the largest element (1e-4)."""
import numpy as np
import pytest

import oracle as O
import vie_synth as V

torch = pytest.importorskip("torch")
import paper_1610_00835_gb300 as P  # noqa: E402
from gpu_util import dev, host, rel_l2  # noqa: E402

pytestmark = pytest.mark.gpu


def gpu_apply(h, g):
    y = torch.empty(h.N, dtype=torch.float64, device="cuda:0")
    P.vie_apply(h, P.VIE_OP_K_SIGMA_S, dev(g), y, 1)
    return host(y)


def check(dim, n, m, rows):
    g = np.random.default_rng(n).random(m.N) + 0.5
    h = P.vie_create(dim, n, m.sigma_t, m.sigma_s)
    assert P.vie_get_kernel(h) == P.VIE_KERNEL_DISPLACEMENT
    got = gpu_apply(h, g)
    ref = gpu_apply(P.vie_create(dim, n, m.sigma_t, m.sigma_s, kernel=P.VIE_KERNEL_SYMMETRIC), g)
    assert rel_l2(got, ref) < 2e-5
    assert np.max(np.abs(got - ref)) < 1e-4 * np.max(np.abs(ref))
    want = O.apply(dim, m.sigma_t, m.sigma_s, g, rows=rows)
    assert rel_l2(got[rows], want) < 1e-5
    np.testing.assert_array_equal(gpu_apply(h, g), got)


# two tiles per unit from n = 96 on; compiled pitches per class of n; from n = 234
# on two windows of the lattice in shared memory, the rest from global memory
@pytest.mark.parametrize("n", [32, 33, 64, 65, 95, 96, 97, 128, 129, 140, 141, 161, 162, 233, 234, 235, 247, 258])
def test_2d_tiles(n):
    m = V.heterogeneous_2d(n=n, seed=31)
    rows = np.unique(np.r_[0, n - 1, m.N - 1, np.random.default_rng(n).integers(0, m.N, 13)])
    check(2, n, m, rows)


# lattice pitch 17 up to n = 16, 33 above; lane extents of every width, 1 to 4 stack blocks
@pytest.mark.parametrize("n", [2, 7, 8, 9, 15, 16, 17, 23, 24, 25, 31, 32])
def test_3d_tiles(n):
    m = V.heterogeneous_3d(n=n, seed=32)
    rows = np.unique(np.r_[0, n - 1, m.N - 1, np.random.default_rng(n).integers(0, m.N, 13)])
    check(3, n, m, rows)
