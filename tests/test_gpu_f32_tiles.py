"""The fast DCT's two CTA sizes: alone a cube's tiles are few (64 threads up to
a number that depends on the bands, 256 where spectra are short or long), in a
batch many (256), and the transforms are the same operations, so a cube has the
same bits either way."""
import numpy as np
import pytest

from synth import fdmc_eps, make_cube
from tests.gpu_util import cuda, dev

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,L,B,sure", [(16, 8, 3, False), (32, 16, 40, True), (32, 32, 40, True),
                                        (32, 128, 12, False), (32, 256, 6, False), (16, 256, 8, True),
                                        (16, 512, 6, False), (8, 512, 12, True), (8, 1024, 4, False)])
def test_fast_dct_batch_has_the_bits_of_a_cube_alone(n, L, B, sure):
    torch = cuda()
    import paper_1905_08468_gb300 as pkg
    c = make_cube(n, L, max(2, n // 4), 1, 30 * n, seed=2000 + L)
    kw = dict(window=3, eta=(1e-6, 1e-6), eps=fdmc_eps(c.noise_var))
    x = {b: torch.zeros((b, L, n, n), device="cuda") for b in (1, B)}
    for b in x:
        rep = lambda a: np.stack([a] * b) if b > 1 else a
        with pkg.Plan(n, L, rep(c.psf), sure=sure, n_wavelets=2, levels=1, batch=b, precision="fp32") as p:
            d = dev(rep(c.dirty), torch)
            if sure:
                th = [(0.03, 0.02)] * b if b > 1 else (0.03, 0.02)
                p.sure_tune(d, dev(rep(c.delta), torch), np.concatenate([c.noise_var] * b), x[b], th, 7, **kw)
            else:
                p.solve(d, x[b], 6, [1e-2] * b if b > 1 else 1e-2, [2e-2] * b if b > 1 else 2e-2)
    for i in range(B):
        assert torch.equal(x[B][i], x[1][0]), i


@pytest.mark.parametrize("n,L,J", [(32, 2, 3), (32, 8, 3), (16, 32, 2), (16, 64, 2), (8, 256, 2), (4, 1024, 2)])
def test_default_precision_matches_oracle(n, L, J):
    """The default spectral step of power-of-two band counts (the fast DCT,
    tcgen05 for 64) in a plain solve; cube relative L2 1e-5."""
    torch = cuda()
    import paper_1905_08468_gb300 as pkg
    from oracle import muffin as om
    from tests.gpu_util import host, rel_l2
    c = make_cube(n, L, max(2, n // 4), 1, 30 * n, seed=2100 + L)
    x = torch.zeros((L, n, n), device="cuda")
    with pkg.Plan(n, L, c.psf, n_wavelets=3, levels=J) as p:
        p.solve(dev(c.dirty, torch), x, 20, 1e-2, 2e-2)
    st, _ = om.solve(om.make_problem(c.dirty, c.psf, n_wavelets=3, J=J), 1e-2, 2e-2, 20)
    assert rel_l2(host(x), st.x) <= 1e-5
