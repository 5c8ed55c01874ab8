"""lx3c_boys far beyond the table and beyond the range of the reciprocal root's
single-precision seed, with low mantissa bits set: F_m(T) = Gamma(m + 1/2) / 2
T^-(m + 1/2) there, exact to FP64.  (The lower orders come from the highest
one, so that one must not underflow: the order alone beyond 1e60.)  Tolerance
as in test_boys_device (6e-15: about an ulp for each of the multiplications)."""
import math

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("T,mmax", [(1.7e7, 3), (1e30, 3), (3.3e38, 3), (3.5e38, 3), (1e39, 3), (1e60, 3),
                                    (1e60, 0), (1e150, 0), (1.7e308, 0)])
def test_asymptotic_boys(T, mmax):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2210_03192_gb300 as lx
    g = lx.boys(torch.tensor([T, np.nextafter(T, 0.0)], device="cuda"), mmax).cpu().numpy()
    for m in range(mmax + 1):
        # T^-(m + 1/2) without overflow on the way
        ref = math.exp(math.lgamma(m + 0.5)) / 2 / math.sqrt(T)
        for _ in range(m):
            ref /= T
        assert np.all(np.abs(g[:, m] - ref) <= 6e-15 * ref), (m, g[:, m], ref)
