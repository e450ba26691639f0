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


def on_a_side_stream(call):
    """The call's outputs from a stream of its own while the default one is busy (for about 0.2 s)."""
    torch.cuda.synchronize()
    torch.cuda._sleep(400_000_000)
    side = torch.cuda.Stream()
    out = call(side)
    side.synchronize()
    return host(out)


# one block, a cluster, the whole grid; several sources
@pytest.mark.parametrize("n,R", [(12, 1), (64, 1), (136, 1), (64, 3), (136, 3)])
def test_solver_workspaces_are_cleared_on_the_stream_of_the_solve(n, R):
    m = V.heterogeneous_2d(n=n, seed=5700)
    f = dev(V.bump_sources(2, n, R, 5701).reshape(-1))

    def solve(stream):
        U = torch.empty_like(f)
        P.vie_solve_gmres(h, f, U, rtol=1e-8, nrhs=R, stream=stream)
        return U

    h = P.vie_create(2, n, m.sigma_t, m.sigma_s)
    want = host(solve(None))
    P.vie_destroy(h)  # (the next handle takes its buffers, with what was in them)
    h = P.vie_create(2, n, m.sigma_t, m.sigma_s)
    np.testing.assert_array_equal(on_a_side_stream(solve), want)


@pytest.mark.parametrize("channels", [32, 16])
def test_network_workspaces_are_cleared_on_the_stream_of_the_call(channels):
    n, B = 32, 2
    x = dev(np.random.default_rng(5).standard_normal(B * 3 * n * n), torch.float32)

    def forward(stream):
        o = torch.empty(B * n * n, dtype=torch.float32, device="cuda:0")
        P.vie_unet_forward(net, x, o, B, n, use_bf16=True, stream=stream)
        return o

    net = P.vie_unet_create(3, channels, seed=6)
    want = host(forward(None))
    P.vie_unet_destroy(net)
    net = P.vie_unet_create(3, channels, seed=6)
    np.testing.assert_array_equal(on_a_side_stream(forward), want)
