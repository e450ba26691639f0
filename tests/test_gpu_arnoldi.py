"""The one-launch Arnoldi step in each of its forms: one block, a cluster, the whole grid, w in registers or not."""
import numpy as np
import pytest

import vie_synth as V

torch = pytest.importorskip("torch")
import paper_1610_00835_gb300 as P  # noqa: E402
from gpu_util import host  # noqa: E402

pytestmark = pytest.mark.gpu


# cells: 144 (one block), 4096 (16 blocks of one element a thread), 16384 (four), 36864 (36 blocks), 331776 (304, w in memory)
@pytest.mark.parametrize("n,fmm", [(12, False), (64, False), (128, True), (192, True), (576, True)])
@pytest.mark.parametrize("restart", [64, 5])
def test_solution_has_the_reported_residual(n, fmm, restart):
    m = V.homogeneous_medium(2, n, 20.2, 20.0)  # slow convergence: more than eight basis vectors
    kw = {} if fmm else {"precision": P.VIE_PREC_FP64}
    h = P.vie_create(2, n, m.sigma_t, m.sigma_s, tau_mode=P.VIE_TAU_CLOSED, **kw)
    if fmm:
        P.vie_assemble_fmm(h, 4)
    f = torch.as_tensor(m.f, dtype=torch.float64, device="cuda:0")
    U, phi, r = torch.empty_like(f), torch.empty_like(f), torch.empty_like(f)
    rtol = 1e-5 if fmm else 1e-11  # the FP32 operator of this medium leaves 7e-7 at 576^2
    rep = P.vie_solve_gmres(h, f, U, rtol=rtol, restart=restart)
    assert rep["converged"] and rep["iters"] > 8
    P.vie_apply(h, P.VIE_OP_A_RAW, f, phi)
    P.vie_apply(h, P.VIE_OP_I_MINUS_K, U, r)
    res = float((phi - r).norm() / phi.norm())
    # the solver's own true residual, recomputed: rounding of the subtraction alone
    assert res <= rtol * (1 + 1e-6) and abs(res - rep["relres"]) <= 1e-6 * rtol + 1e-15
    if not fmm:
        # within a cycle the estimate is the residual (orthogonal basis, right rotations); an FP32 operator rounds
        # every basis vector it is applied to, which the estimate does not see
        assert abs(rep["relres_est"] - rep["relres"]) <= 0.01 * rtol


@pytest.mark.parametrize("n", [20, 136])  # a cluster per source; more blocks than a cluster holds
def test_lockstep_solutions_equal_single_ones(n):
    m = V.heterogeneous_2d(n=n)
    h = P.vie_create(2, n, m.sigma_t, m.sigma_s)
    F = V.bump_sources(2, n, 3, 90 + n)
    f = torch.as_tensor(F, dtype=torch.float64, device="cuda:0")
    U = torch.empty(3 * m.N, dtype=torch.float64, device="cuda:0")
    P.vie_solve_gmres(h, f.reshape(-1), U, rtol=1e-8, nrhs=3)
    for r in range(3):
        u = torch.empty(m.N, dtype=torch.float64, device="cuda:0")
        P.vie_solve_gmres(h, f[r].contiguous(), u, rtol=1e-8)
        np.testing.assert_array_equal(host(U).reshape(3, -1)[r], host(u))
