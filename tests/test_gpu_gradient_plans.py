"""Gradient FFT passes at the sizes where the plans change: two and three
stages of the in-place column plan with every last radix, the first row stage
and the last one in registers or through shared memory, ragged last column
groups, both radices.  Tolerance: the gradient operator's relative L2 1e-6."""
import numpy as np
import pytest

from oracle import convolution
from tests.gpu_util import cuda, dev, host, rel_l2

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,L", [(2, 2), (16, 3), (32, 5), (64, 3), (128, 2), (256, 1), (512, 2),
                                 (1024, 1), (2048, 1)])
@pytest.mark.parametrize("radix", [16, 8])
def test_gradient(n, L, radix):
    torch = cuda()
    import paper_1905_08468_gb300 as pkg
    rng = np.random.default_rng(n + radix)
    psf = rng.normal(0, 0.05, (L, n, n)).astype(np.float32)
    psf[:, 0, 0] = 1.0
    x, y = rng.standard_normal((2, L, n, n)).astype(np.float32)
    hh = convolution.psf_spectrum(psf)
    ref = convolution.HT(convolution.H(x.astype(np.float64), hh) - y.astype(np.float64), hh)
    g = torch.full((L, n, n), float("nan"), device="cuda")
    with pkg.Plan(n, L, psf, levels=0, n_wavelets=1) as p:
        p.set_schedule(fft_radix=radix)
        p.op_gradient(dev(x, torch), g, dirty=dev(y, torch))
    assert rel_l2(host(g), ref) <= 1e-6
