"""The sweep far behind an absorber: what is left of a source tens of optical depths away, to FP32's own accuracy.

A constant sigma_t and directions along axes make tau exact (multiples of 1/2), so what remains is the transmission
(expf: 2 ulp, 2.4e-7), the step's factor (polynomial, a product: 1.8e-7), the product with Q and the sum over the three steps
that meet the source (2.4e-7): 6.6e-7 relative, 8e-7 allowed.  An exponential that rounds tau log2(e) once loses 2.6e-6."""
import numpy as np
import pytest

import oracle as O

torch = pytest.importorskip("torch")
import paper_1610_00835_gb300 as P  # noqa: E402
from gpu_util import dev, host  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dim,n", [(2, 64), (2, 128), (3, 32)])
def test_transmission_of_thick_media(dim, n):
    N, sigma = n ** dim, float(min(64, n))  # (a step of half a cell has an optical depth of at most 1/2)
    st = np.full(N, sigma)
    for axis in range(dim):
        f = (np.arange(N) // n ** axis % n == 0).astype(np.float64)  # the layer of cells at the boundary
        v = np.eye(dim)[axis:axis + 1]
        h = P.vie_create(dim, n, st, np.zeros(N))
        Phi = torch.empty(N, dtype=torch.float32, device="cuda:0")
        P.ert_sweep(h, dev(np.zeros(N)), dev(f), torch.as_tensor(v.astype(np.float32), device="cuda:0"), Phi)
        want = O.sweep(dim, st, f, v)[0]
        assert want.min() < 1e-12
        np.testing.assert_allclose(host(Phi), want, rtol=8e-7, atol=0)
