"""H^T y is formed on pairs of FP32 values (48 bits) and rounded to FP32 once:
every pixel is the 64-bit result's rounding to within what 48-bit transforms
leave.  Bound, element by element: half a unit in the last place (2^-24 of the
value), plus the transforms' rounding, two of 2 log2 n <= 22 levels whose errors
of at most 2^-46 of the image's largest value a level add up to less than
2^-40 of it (an FP32 transform would be off by 2^-24 of it)."""
import numpy as np
import pytest

from oracle import convolution
from tests.gpu_util import cuda, dev, host

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,L", [(16, 5), (64, 6), (256, 3), (2048, 1), (1024, 2)])
@pytest.mark.parametrize("faint", [1.0, 1e-6])
def test_every_pixel_is_rounded_once(n, L, faint):
    torch = cuda()
    import paper_1905_08468_gb300 as pkg
    rng = np.random.default_rng(n + L)
    psf = rng.normal(0, 0.05, (L, n, n)).astype(np.float32)
    psf[:, 0, 0] = 1.0
    y = rng.standard_normal((L, n, n)).astype(np.float32)
    y[1::2] *= np.float32(faint)                       # beside a bright partner
    ref = convolution.HT(y.astype(np.float64), convolution.psf_spectrum(psf))
    g = torch.empty((L, n, n), device="cuda")
    with pkg.Plan(n, L, psf, n_wavelets=1, levels=0) as p:
        p.op_gradient(torch.zeros_like(g), g, dirty=dev(y, torch))
    off = np.abs(-host(g) - ref)
    largest = np.abs(ref).max(axis=(1, 2), keepdims=True)
    assert np.all(off <= 2.0 ** -24 * np.abs(ref) * (1 + 2.0 ** -20) + 2.0 ** -40 * largest)
