"""A batch's graph replays the kernels of its media's own applies, and counts them."""
import numpy as np
import pytest

import vie_synth as V

torch = pytest.importorskip("torch")
import paper_1610_00835_gb300 as P  # noqa: E402
from gpu_util import dev  # noqa: E402

pytestmark = pytest.mark.gpu


def launches(call):
    before = P.vie_kernel_launches()
    call()
    return P.vie_kernel_launches() - before


# one march up to 233, three (two windows of the lattice and the rest) from 234 on
@pytest.mark.parametrize("ns", [(24,), (233,), (234,), (258, 24)])
def test_replays_count_every_launch(ns):
    media = [V.heterogeneous_2d(n=n, seed=n) for n in ns]
    b = P.vie_batch_create(list(ns), [m.sigma_t for m in media], [m.sigma_s for m in media])
    g = dev(np.concatenate([m.f for m in media]))
    y = torch.empty_like(g)
    run = lambda: P.vie_batch_apply(b, P.VIE_OP_K_SIGMA_S, g, y)  # noqa: E731
    run()  # (captures the graph)
    single = 0
    for m in media:
        h = P.vie_create(2, m.n, m.sigma_t, m.sigma_s)
        gm = dev(m.f)
        single += launches(lambda: P.vie_apply(h, P.VIE_OP_K_SIGMA_S, gm, torch.empty_like(gm)))
    # the batch adds the source kernel of the media without a march of their own
    assert launches(run) == single + 1
