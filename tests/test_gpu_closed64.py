"""FP64 applies of homogeneous media (closed-form optical depth, entries by displacement) against the oracle."""
import numpy as np
import pytest

import oracle as O

torch = pytest.importorskip("torch")
import paper_1610_00835_gb300 as P  # noqa: E402
from gpu_util import dev, host, rel_l2  # noqa: E402

pytestmark = pytest.mark.gpu


def applied(dim, n, st, ss, g, op):
    h = P.vie_create(dim, n, st, ss, tau_mode=P.VIE_TAU_CLOSED, precision=P.VIE_PREC_FP64)
    y = torch.empty(n ** dim, dtype=torch.float64, device="cuda:0")
    P.vie_apply(h, op, dev(g), y)
    return host(y)


# one cell; fewer rows than a thread stacks; ragged last row block; more than one CTA of targets; 3D
@pytest.mark.parametrize("dim,n,sigma", [(2, 1, 2.0), (2, 2, 0.0), (2, 3, 1.1), (2, 5, 40.0), (2, 33, 3.0),
                                         (2, 50, 1.1), (3, 1, 1.0), (3, 2, 0.0), (3, 5, 9.0), (3, 9, 1.3)])
@pytest.mark.parametrize("op", [P.VIE_OP_K_SIGMA_S, P.VIE_OP_I_MINUS_K, P.VIE_OP_A_RAW])
def test_closed_entries_match_oracle(dim, n, sigma, op):
    N = n ** dim
    rng = np.random.default_rng([dim, n])
    st, ss, g = np.full(N, sigma), rng.uniform(0.0, 1.0, N), rng.standard_normal(N)
    want = O.apply(dim, st, ss, g, op=op, mode=O.TAU_CLOSED)
    assert rel_l2(applied(dim, n, st, ss, g, op), want) < 1e-12  # the FP64 path's bar


def test_infinite_and_nan_sources_stay_what_they_are():
    n = 18
    st, ss = np.full(n * n, 1.0), np.ones(n * n)
    g = np.ones(n * n)
    g[100] = np.inf
    y = applied(2, n, st, ss, g, P.VIE_OP_A_RAW)
    assert np.all(np.isposinf(y))  # the own cell enters through the diagonal alone, not as 0 * inf
    g[100] = np.nan
    assert np.all(np.isnan(applied(2, n, st, ss, g, P.VIE_OP_A_RAW)))
