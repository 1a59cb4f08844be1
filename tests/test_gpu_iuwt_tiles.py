"""Starlet kernels at the edges of their 32 x 128 tiles: images smaller than a
tile, one and two tiles wide, the widest halo (four scales) and one scale only,
three chains (masks handed from the primal's launch to the derivatives')
against the oracle.  Tolerances as the starlet's other tests: operators 1e-6,
cube 1e-5, theta 1e-3."""
import numpy as np
import pytest

from oracle import iuwt, muffin as om, sure as osu
from synth import fdmc_eps, make_cube
from tests.gpu_util import cuda, dev, host, rel_l2

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,L,J", [(2, 2, 1), (16, 1, 4), (256, 2, 4), (512, 1, 1)])
def test_operators(n, L, J):
    torch = cuda()
    import paper_1905_08468_gb300 as pkg
    rng = np.random.default_rng(n + J)
    psf = np.zeros((L, n, n), np.float32)
    psf[:, 0, 0] = 1.0
    x = rng.normal(size=(L, n, n)).astype(np.float32)
    u = rng.normal(size=(L, J + 1, n, n)).astype(np.float32)
    uo = torch.full((L, J + 1, n, n), float("nan"), device="cuda")
    xo = torch.full((L, n, n), float("nan"), device="cuda")
    with pkg.Plan(n, L, psf, levels=J, dictionary="iuwt") as p:
        p.op_analysis(dev(x, torch), uo)
        p.op_synthesis(dev(u, torch), xo)
    assert rel_l2(host(uo), iuwt.analysis(x.astype(np.float64), J)) <= 1e-6
    assert rel_l2(host(xo), iuwt.adjoint(u.astype(np.float64), J)) <= 1e-6


@pytest.mark.parametrize("n,L,J", [(8, 3, 1), (16, 2, 4), (128, 2, 2), (256, 1, 4)])
def test_three_chains(n, L, J):
    torch = cuda()
    import paper_1905_08468_gb300 as pkg
    c = make_cube(n, L, max(3, n // 4), 1, max(400, 30 * n), seed=1500 + n)
    eps, eta = fdmc_eps(c.noise_var), (0.2 / c.voxels, 2.0 / c.voxels)
    x = torch.zeros((L, n, n), device="cuda")
    with pkg.Plan(n, L, c.psf, levels=J, dictionary="iuwt", sure=True) as p:
        th, _, _ = p.sure_tune(dev(c.dirty, torch), dev(c.delta, torch), c.noise_var, x,
                               (0.03, 0.02), 12, window=4, eta=eta, eps=eps)
    prob = om.make_problem(c.dirty, c.psf, J=J, dictionary="iuwt")
    r = osu.ada_pt(prob, c.delta, eps, c.noise_var, (0.03, 0.02), 12, Delta=4, eta=eta)
    assert rel_l2(host(x), r.x) <= 1e-5
    assert np.max(np.abs(np.array(th) / r.theta - 1)) <= 1e-3
