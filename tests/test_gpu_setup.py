"""Set-up transforms that carry two bands of a cube in one complex image: odd
and even band counts, several cubes, bands whose images or PSFs differ by many
orders of magnitude, and a band with a NaN beside a finite one.  Tolerance: the
gradient operator's relative L2 1e-6, band by band."""
import numpy as np
import pytest

from oracle import convolution
from tests.gpu_util import cuda, dev, host, rel_l2

pytestmark = pytest.mark.gpu


def problem(n, bands, seed):
    rng = np.random.default_rng(seed)
    psf = rng.normal(0, 0.05, (bands, n, n)).astype(np.float32)
    psf[:, 0, 0] = 1.0
    return psf, rng.standard_normal((bands, n, n)).astype(np.float32)


@pytest.mark.parametrize("n,L,B", [(2, 1, 1), (8, 2, 1), (32, 3, 2), (64, 5, 1), (2048, 2, 1)])
@pytest.mark.parametrize("spread", [0, 12])
def test_adjoint_of_every_band(n, L, B, spread):
    """g = -H^T y at x = 0, bands of a pair up to 10^spread apart."""
    torch = cuda()
    import paper_1905_08468_gb300 as pkg
    psf, y = problem(n, L * B, 11 * n + L)
    scale = 10.0 ** (spread * (np.arange(L * B) % 2 - 0.5))
    y = (y * scale[:, None, None]).astype(np.float32)
    psf = (psf * scale[::-1, None, None] ** 0.5).astype(np.float32)
    ref = -convolution.HT(y.astype(np.float64), convolution.psf_spectrum(psf))
    g = torch.empty((L * B, n, n), device="cuda")
    with pkg.Plan(n, L, psf, batch=B, levels=0) as p:
        p.op_gradient(torch.zeros_like(g), g, dirty=dev(y, torch))
        beta = np.atleast_1d(p.lipschitz)
    for l in range(L * B):
        assert rel_l2(host(g[l]), ref[l]) <= 1e-6, l
    power = np.abs(np.fft.fft2(psf.astype(np.float64))) ** 2
    assert np.allclose(beta, power.reshape(B, -1).max(1), rtol=1e-12)


def test_nan_band_leaves_its_pair_alone():
    torch = cuda()
    import paper_1905_08468_gb300 as pkg
    n, L = 32, 4
    psf, y = problem(n, L, 3)
    ref = -convolution.HT(y.astype(np.float64), convolution.psf_spectrum(psf))
    y[2, 5, 7] = np.nan
    g = torch.empty((L, n, n), device="cuda")
    with pkg.Plan(n, L, psf) as p:
        p.op_gradient(torch.zeros_like(g), g, dirty=dev(y, torch))
    assert torch.isnan(g[2]).all()
    for l in (0, 1, 3):
        assert rel_l2(host(g[l]), ref[l]) <= 1e-6


def test_objective_of_bands_apart_and_negative_cube():
    """The FP64 residual with odd bands and the indicator of the positive
    orthant; tolerance 1e-6 as the objective's other tests."""
    torch = cuda()
    import paper_1905_08468_gb300 as pkg
    from oracle import muffin as om
    n, L = 32, 3
    psf, y = problem(n, L, 9)
    y[1] *= 1e3
    x = np.abs(problem(n, L, 10)[1])
    with pkg.Plan(n, L, psf) as p:
        f = p.objective(dev(y, torch), dev(x, torch), 0.02, 0.03)
        x[2, 1, 1] = -1e-3
        assert np.isinf(p.objective(dev(y, torch), dev(x, torch), 0.02, 0.03))
        x[2, 1, 1] = -0.0
        assert np.isfinite(p.objective(dev(y, torch), dev(x, torch), 0.02, 0.03))
        x[2, 1, 1] = np.abs(problem(n, L, 10)[1])[2, 1, 1]
    prob = om.make_problem(y, psf)
    assert f == pytest.approx(om.objective(x.astype(np.float64), prob, 0.02, 0.03), rel=1e-6)
