"""An Arnoldi vector whose squared norm overflows ends the solve in its step, before anything reaches the solution."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
import paper_1610_00835_gb300 as P  # noqa: E402
from gpu_util import dev, host  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,nrhs", [(8, 1), (40, 1), (130, 1), (8, 2), (130, 2)])
def test_overflow_of_a_norm_is_reported_by_its_step(n, nrhs):
    N = n * n
    st, ss = np.full(N, 1.0), np.full(N, 0.5)
    ss[N // 2] = 1e160  # entries of K v up to about 1e156 or more, their squares past 1.8e308
    h = P.vie_create(2, n, st, ss, tau_mode=P.VIE_TAU_CLOSED, precision=P.VIE_PREC_FP64)
    U = torch.zeros(nrhs * N, dtype=torch.float64, device="cuda:0")
    with pytest.raises(P.VieError, match="non-finite Arnoldi step") as e:
        P.vie_solve_gmres(h, dev(np.random.default_rng(n).random(nrhs * N)), U, nrhs=nrhs)
    assert e.value.status == P.vie.VIE_ERR_NONFINITE
    assert np.all(host(U) == 0.0)
