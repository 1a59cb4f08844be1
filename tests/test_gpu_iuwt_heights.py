"""The starlet kernels' two tile heights: one cube runs tiles of 8 rows, a batch
of enough of them (a wave of 32-row tiles) the high ones, with the same sums in
the same order, so a cube's result is the same bits either way.  Images smaller
than a tile, one tile and several tiles wide, the narrowest and the widest halo;
the single cube against the oracle."""
import numpy as np
import pytest

from oracle import iuwt, muffin as om
from synth import fdmc_eps, make_cube
from tests.gpu_util import cuda, dev, host, rel_l2

pytestmark = pytest.mark.gpu

# n, bands, scales, cubes: ceil(n / 128) ceil(n / 32) bands cubes >= 456 tiles of 32 rows
SHAPES = [(4, 5, 2, 92), (16, 6, 4, 76), (64, 3, 1, 76), (64, 3, 4, 76), (256, 2, 3, 15)]


def cubes(n, L):
    return [make_cube(n, L, max(2, n // 4), 1, max(200, 30 * n), seed=1700 + n + i) for i in range(2)]


@pytest.mark.parametrize("n,L,J,B", SHAPES)
def test_plain_and_operators(n, L, J, B):
    torch = cuda()
    import paper_1905_08468_gb300 as pkg
    cs = cubes(n, L)
    u0 = np.random.default_rng(n).normal(size=(2, L, J + 1, n, n)).astype(np.float32)
    one = []
    for c, u in zip(cs, u0):
        x, a, s = (torch.zeros(k, device="cuda") for k in ((L, n, n), (L, J + 1, n, n), (L, n, n)))
        with pkg.Plan(n, L, c.psf, levels=J, dictionary="iuwt") as p:
            p.solve(dev(c.dirty, torch), x, 10, 1e-2, 2e-2)
            p.op_analysis(dev(c.dirty, torch), a)
            p.op_synthesis(dev(u, torch), s)
        assert rel_l2(host(a), iuwt.analysis(c.dirty.astype(np.float64), J)) <= 1e-6
        assert rel_l2(host(s), iuwt.adjoint(u.astype(np.float64), J)) <= 1e-6
        st, _ = om.solve(om.make_problem(c.dirty, c.psf, J=J, dictionary="iuwt"), 1e-2, 2e-2, 10)
        assert rel_l2(host(x), st.x) <= 1e-5
        one.append((x, a, s))
    pick = [i % 2 for i in range(B)]
    stack = lambda v: dev(np.stack([v[i] for i in pick]), torch)
    x, a, s = (torch.zeros(k, device="cuda") for k in ((B, L, n, n), (B, L, J + 1, n, n), (B, L, n, n)))
    with pkg.Plan(n, L, stack([c.psf for c in cs]), levels=J, dictionary="iuwt", batch=B) as p:
        d = stack([c.dirty for c in cs])
        p.solve(d, x, 10, [1e-2] * B, [2e-2] * B)
        p.op_analysis(d, a)
        p.op_synthesis(stack(u0), s)
    for i, k in enumerate(pick):
        for got, want in zip((x, a, s), one[k]):
            assert torch.equal(got[i], want), i


@pytest.mark.parametrize("n,L,J,B", [SHAPES[1], SHAPES[3], SHAPES[4]])
def test_three_chains(n, L, J, B):
    torch = cuda()
    import paper_1905_08468_gb300 as pkg
    cs = cubes(n, L)
    kw = dict(window=3, eta=(1e-6, 1e-6), eps=fdmc_eps(cs[0].noise_var))
    one = []
    for c in cs:
        x = torch.zeros((L, n, n), device="cuda")
        with pkg.Plan(n, L, c.psf, levels=J, dictionary="iuwt", sure=True) as p:
            th, _, _ = p.sure_tune(dev(c.dirty, torch), dev(c.delta, torch), c.noise_var, x,
                                   (0.03, 0.02), 7, **kw)
        one.append((x, th))
    pick = [i % 2 for i in range(B)]
    stack = lambda v: dev(np.stack([v[i] for i in pick]), torch)
    x = torch.zeros((B, L, n, n), device="cuda")
    with pkg.Plan(n, L, stack([c.psf for c in cs]), levels=J, dictionary="iuwt", batch=B, sure=True) as p:
        th, _, _ = p.sure_tune(stack([c.dirty for c in cs]), stack([c.delta for c in cs]),
                               np.concatenate([cs[i].noise_var for i in pick]), x, [(0.03, 0.02)] * B, 7, **kw)
    for i, k in enumerate(pick):
        assert torch.equal(x[i], one[k][0]) and tuple(th[i]) == tuple(one[k][1]), i
