"""PSFs that are not finite: one with an infinite entry has an infinite spectrum
and is refused (EINVAL), whatever the other bands hold; one with a NaN is
passed over beside a finite band, and refused alone."""
import numpy as np
import pytest

from tests.gpu_util import cuda

pytestmark = pytest.mark.gpu

N, L = 32, 3


def psfs(bands=L):
    psf = np.random.default_rng(5).normal(0, 0.05, (bands, N, N)).astype(np.float32)
    psf[:, 0, 0] = 1.0
    return psf


@pytest.mark.parametrize("band", [0, 1, 2])
@pytest.mark.parametrize("at,value", [((0, 0), np.inf), ((0, 0), -np.inf), ((3, 5), np.inf)])
def test_infinite_psf_is_refused(band, at, value):
    cuda()
    import paper_1905_08468_gb300 as pkg
    good = psfs()
    bad = good.copy()
    bad[band][at] = value
    with pytest.raises(pkg.MuffinError) as e:
        pkg.Plan(N, L, bad, n_wavelets=1, levels=1)
    assert e.value.status == 1
    with pkg.Plan(N, L, good, n_wavelets=1, levels=1) as p:
        beta = p.lipschitz
        with pytest.raises(pkg.MuffinError) as e:
            p.load_psf(bad)
        assert e.value.status == 1
        p.load_psf(good)                             # the plan stays usable
        assert p.lipschitz == beta
    two = np.stack([good, bad])
    with pytest.raises(pkg.MuffinError) as e:        # the second cube of a batch
        pkg.Plan(N, L, two, n_wavelets=1, levels=1, batch=2)
    assert e.value.status == 1


def test_server_rejects_an_infinite_psf():
    cuda()
    import paper_1905_08468_gb300 as pkg
    bad = psfs()
    bad[1, 0, 0] = np.inf
    with pkg.Server(max_batch=2, chunk=5) as srv:
        t = srv.submit(bad, np.ones((L, N, N), np.float32), 1e-2, 1e-2, 5)
        with pytest.raises(pkg.MuffinError) as e:
            for _ in range(20):
                srv.step()
                if srv.poll(t, np.empty((L, N, N), np.float32)):
                    break                            # served: no error
        assert e.value.status == 1


def test_nan_psf_as_before():
    cuda()
    import paper_1905_08468_gb300 as pkg
    psf = psfs()
    psf[1, 4, 4] = np.nan
    beta = (np.abs(np.fft.fft2(psf[[0, 2]].astype(np.float64))) ** 2).max()
    with pkg.Plan(N, L, psf, n_wavelets=1, levels=1) as p:
        assert np.isclose(p.lipschitz, beta, rtol=1e-12)
    with pytest.raises(pkg.MuffinError) as e:
        pkg.Plan(N, 1, psf[1:2], n_wavelets=1, levels=1)
    assert e.value.status == 1
