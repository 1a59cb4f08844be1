"""Spectral step at the edges of its kernels' ranges: the dense folded
products (odd and even band counts, the change of task size at 40 bands, one
band, more bands than a 64-pixel tile holds) and the fast DCT with 64-thread
CTAs, both on pixel blocks that start anywhere (the sharded form)."""
import ctypes

import numpy as np
import pytest

from tests.gpu_util import cuda, dev, host, rel_l2

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("L", [1, 2, 3, 32, 39, 40, 41, 130, 256, 351])
@pytest.mark.parametrize("p0", [0, 3])
def test_shard_step_any_bands_and_block(L, p0):
    """v = sat(v + sigma gamma alpha C z), t = gamma alpha C^T v against the
    dense product in 64 bits.  Tolerance: FP32 sums of at most 128 folded
    terms, 2e-6 as the DCT operator's."""
    torch = cuda()
    import paper_1905_08468_gb300 as pkg
    from oracle import spectral
    from paper_1905_08468_gb300 import native
    n, npix, gamma, sigma = 16, 64 * 3 + 4, 0.7, 10.0
    rng = np.random.default_rng(100 * L + p0)
    alpha = rng.uniform(0.05, 0.15, (n, n)).astype(np.float32)
    psf = np.zeros((L, n, n), np.float32)
    psf[:, 0, 0] = 1
    z, v = (rng.normal(0, s, (L, npix)).astype(np.float32) for s in (1.0, 0.5))
    zt, vt = dev(z, torch), dev(v, torch)
    tt = torch.full_like(zt, 7.0)
    with pkg.Plan(n, L, psf, n_wavelets=1, levels=1, alpha=alpha) as p:
        native.check(p._lib.muffin_shard_spectral(
            p._h, *(ctypes.c_void_p(q.data_ptr()) for q in (zt, vt, tt)),
            ctypes.c_int64(p0), ctypes.c_int64(npix), ctypes.c_double(gamma)))
    C = spectral.dct_matrix(L)
    a = alpha.reshape(-1)[p0: p0 + npix].astype(np.float64)
    vr = np.clip(v + sigma * gamma * a * (C @ z.astype(np.float64)), -1, 1)
    assert rel_l2(host(vt), vr) <= 2e-6
    assert rel_l2(host(tt), gamma * a * (C.T @ vr)) <= 2e-6


@pytest.mark.parametrize("L", [3, 40, 66, 351])
def test_three_chains_match_oracle(L):
    """ADA-PT (masks shared by the chains) on the dense kernel."""
    from tests.test_gpu_states import run_case
    from synth import make_cube
    c = make_cube(8, L, 3, 1, 400, seed=700 + L)
    run_case(c, (0.05, 0.05), 8, 3, (1e-6, 1e-5))
