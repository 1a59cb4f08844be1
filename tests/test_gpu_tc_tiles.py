"""Tiles of the 64-band spectral step dealt to CTAs: a partial tile, fewer tiles
than SMs, between one and two an SM, several a group.  A cube's result does not
depend on which CTA and group took its tiles, nor on the cubes beside it, so a
batched solve equals the single ones bit for bit; against the FP32 kernel the
relative L2 bound of the iteration's parity, 1e-5."""
import pytest

from tests.gpu_util import cuda, rel_l2

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,batch", [(8, 3), (32, 2), (128, 2), (256, 3)])
def test_tiles(n, batch):
    torch = cuda()
    import paper_1905_08468_gb300 as pkg
    gen = torch.Generator(device="cuda").manual_seed(n + batch)
    y = torch.rand(batch, 64, n, n, device="cuda", generator=gen)
    psf = torch.zeros(64, n, n, device="cuda")
    psf[:, 0, 0], psf[:, 0, 1] = 1.0, 0.5
    kw = dict(levels=1, n_wavelets=1)
    x = torch.zeros_like(y)
    with pkg.Plan(n, 64, psf.repeat(batch, 1, 1, 1), batch=batch, **kw) as p:
        p.solve(y, x, 4, 1e-2, 2e-2)
    for i in range(batch):
        one, f32 = torch.zeros_like(y[i]), torch.zeros_like(y[i])
        with pkg.Plan(n, 64, psf, **kw) as p:
            p.solve(y[i], one, 4, 1e-2, 2e-2)
        with pkg.Plan(n, 64, psf, precision="fp32", **kw) as p:
            p.solve(y[i], f32, 4, 1e-2, 2e-2)
        torch.cuda.synchronize()
        assert float(one.norm()) > 0
        assert torch.equal(x[i], one)
        assert rel_l2(one.cpu().numpy(), f32.cpu().numpy()) <= 1e-5
