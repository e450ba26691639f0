"""A grid-wide barrier of the Arnoldi step that runs out: the solve says so, and the next one is the same as ever."""
import numpy as np
import pytest

import vie_synth as V

torch = pytest.importorskip("torch")
import paper_1610_00835_gb300 as P  # noqa: E402
from gpu_util import dev, host  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [129, 192])  # 17 blocks, 36 blocks
def test_barrier_timeout_is_reported_then_the_next_solve_runs(n):
    m = V.heterogeneous_2d(n=n, seed=5800)
    f = dev(m.f)
    U = torch.empty_like(f)
    P.vie_solve_gmres(P.vie_create(2, n, m.sigma_t, m.sigma_s), f, U, rtol=1e-8)
    want = host(U)
    h = P.vie_create(2, n, m.sigma_t, m.sigma_s)
    try:
        P.vie_set_wait_limits(1000.0, 0.0)
        for _ in range(2):
            with pytest.raises(P.VieError) as e:
                P.vie_solve_gmres(h, f, U, rtol=1e-8)
            assert e.value.status == P.VIE_ERR_TIMEOUT
    finally:
        P.vie_set_wait_limits(1000.0, -1.0)
    assert P.vie_solve_gmres(h, f, U, rtol=1e-8)["converged"]
    np.testing.assert_array_equal(host(U), want)
