"""The forms of the dense spectral kernel that depend on how many pixels there
are: tiles of 16, 32 and 64 pixels, the persistent grid that walks several
tiles a CTA, the number of threads and of rows a task.  All of them compute the
same sums in the same order, so a cube in a batch (many tiles) has the bits that
it has alone (few), and every grid gives the same bits; the sharded form on a
large ragged block and the single cubes are compared with the oracle.
Tolerances as the kernel's other tests."""
import ctypes

import numpy as np
import pytest

from oracle import muffin as om, spectral
from synth import fdmc_eps, make_cube
from tests.gpu_util import cuda, dev, host, rel_l2

pytestmark = pytest.mark.gpu

W32, W64 = 32 * 304 + 4, 64 * 304 + 4       # pixels: tiles of 32, of 64, the last one ragged


@pytest.mark.parametrize("L,npix", [(1, W64), (3, W32), (37, W32), (37, W64), (41, W64), (66, W32),
                                    (130, W64), (199, W32), (200, W32), (250, W64), (259, 516),
                                    (260, 516), (299, 516), (300, W32), (351, 516)])
def test_wide_tiles_match_oracle(L, npix):
    torch = cuda()
    import paper_1905_08468_gb300 as pkg
    from paper_1905_08468_gb300 import native
    n, gamma, sigma, p0 = 256, 0.7, 10.0, 5
    rng = np.random.default_rng(L + npix)
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


# n, bands, cubes: alone 16-pixel tiles, in the batch 32- or 64-pixel ones
BATCHES = [(64, 20, 3), (64, 20, 5), (64, 48, 3), (64, 48, 5), (32, 101, 10), (32, 230, 20)]


@pytest.mark.parametrize("n,L,B", BATCHES)
def test_batch_has_the_bits_of_a_cube_alone(n, L, B):
    torch = cuda()
    import paper_1905_08468_gb300 as pkg
    cs = [make_cube(n, L, n // 4, 1, 30 * n, seed=1900 + L + i) for i in range(2)]
    one = []
    for c in cs:
        x, v, w = (torch.zeros((L, n, n), device="cuda") for _ in range(3))
        with pkg.Plan(n, L, c.psf, n_wavelets=2, levels=1) as p:
            p.solve(dev(c.dirty, torch), x, 6, 1e-2, 2e-2)
            p.op_dct(dev(c.dirty, torch), v)
            p.op_dct(dev(c.dirty, torch), w, inverse=True)
        st, _ = om.solve(om.make_problem(c.dirty, c.psf, n_wavelets=2, J=1), 1e-2, 2e-2, 6)
        assert rel_l2(host(x), st.x) <= 1e-5
        C = spectral.dct_matrix(L)
        assert rel_l2(host(v), spectral.apply_spectra(C, c.dirty.astype(np.float64))) <= 1e-6
        assert rel_l2(host(w), spectral.apply_spectra(C.T, c.dirty.astype(np.float64))) <= 1e-6
        one.append((x, v, w))
    pick = [i % 2 for i in range(B)]
    x, v, w = (torch.zeros((B, L, n, n), device="cuda") for _ in range(3))
    with pkg.Plan(n, L, np.stack([cs[i].psf for i in pick]), n_wavelets=2, levels=1, batch=B) as p:
        d = dev(np.stack([cs[i].dirty for i in pick]), torch)
        p.solve(d, x, 6, [1e-2] * B, [2e-2] * B)
        p.op_dct(d, v)
        p.op_dct(d, w, inverse=True)
    for i, k in enumerate(pick):
        for got, want in zip((x, v, w), one[k]):
            assert torch.equal(got[i], want), i


@pytest.mark.parametrize("n,L,B", [(64, 20, 3), (64, 20, 5), (64, 48, 5), (32, 65, 10)])
def test_three_chains_batch_and_grids(n, L, B):
    """ADA-PT alone (narrow tiles), in a batch (wide ones), and on persistent
    grids of one and two CTAs an SM, each CTA with several tiles."""
    torch = cuda()
    import paper_1905_08468_gb300 as pkg
    c = make_cube(n, L, n // 4, 1, 30 * n, seed=1950 + L)
    kw = dict(window=3, eta=(1e-6, 1e-6), eps=fdmc_eps(c.noise_var))
    x1 = torch.zeros((L, n, n), device="cuda")
    with pkg.Plan(n, L, c.psf, sure=True, n_wavelets=2, levels=1) as p:
        th1, _, _ = p.sure_tune(dev(c.dirty, torch), dev(c.delta, torch), c.noise_var, x1,
                                (0.03, 0.02), 7, **kw)
    for ctas in (0, 1, 2):
        x = torch.zeros((B, L, n, n), device="cuda")
        with pkg.Plan(n, L, np.stack([c.psf] * B), sure=True, n_wavelets=2, levels=1, batch=B) as p:
            p.set_tuning(0, ctas)
            th, _, _ = p.sure_tune(dev(np.stack([c.dirty] * B), torch), dev(np.stack([c.delta] * B), torch),
                                   np.concatenate([c.noise_var] * B), x, [(0.03, 0.02)] * B, 7, **kw)
        for i in range(B):
            assert torch.equal(x[i], x1) and tuple(th[i]) == tuple(th1), (ctas, i)


@pytest.mark.parametrize("n,L", [(128, 20), (128, 37), (128, 66), (128, 201)])
def test_persistent_grids(n, L):
    """More than two tiles an SM, so grids of one and two CTAs an SM loop."""
    torch = cuda()
    import paper_1905_08468_gb300 as pkg
    c = make_cube(n, L, n // 4, 1, 30 * n, seed=1980 + L)
    out = []
    for ctas in (0, 1, 2):
        x = torch.zeros((L, n, n), device="cuda")
        with pkg.Plan(n, L, c.psf, n_wavelets=2, levels=1) as p:
            p.set_tuning(0, ctas)
            p.solve(dev(c.dirty, torch), x, 6, 1e-2, 2e-2)
        out.append(x)
    assert torch.equal(out[1], out[0]) and torch.equal(out[2], out[0])
    if L == 20:
        st, _ = om.solve(om.make_problem(c.dirty, c.psf, n_wavelets=2, J=1), 1e-2, 2e-2, 6)
        assert rel_l2(host(out[0]), st.x) <= 1e-5
