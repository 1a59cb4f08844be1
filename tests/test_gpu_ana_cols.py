"""Analysis levels with the columns of a tile in registers (ana_cols.cu): both
tile heights, one to eight bases, level 1 as the last level and above others,
coarse levels at the kernel's smallest size, and a U that is not 16-byte
aligned (the other kernel), against the oracle's W_s.  Tolerance: the wavelet
operators' relative L2 1e-6."""
import ctypes

import numpy as np
import pytest

from oracle import daubechies, wavelets
from tests.gpu_util import cuda, dev, host, rel_l2

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,L,K,J", [(64, 3, 8, 1), (64, 2, 1, 2), (128, 2, 5, 1), (128, 3, 8, 2),
                                     (256, 2, 3, 2), (256, 1, 8, 3), (1024, 1, 2, 4)])
def test_both_tile_heights_match_oracle(n, L, K, J):
    torch = cuda()
    import paper_1905_08468_gb300 as pkg
    x = np.random.default_rng(n + K).standard_normal((L, n, n)).astype(np.float32)
    psf = np.zeros((L, n, n), np.float32)
    psf[:, 0, 0] = 1.0
    ref = wavelets.Ws(x.astype(np.float64), daubechies.filter_bank(K), J)
    got = []
    for flip in (0, 1):
        u = torch.full((L, K, n, n), float("nan"), device="cuda")
        with pkg.Plan(n, L, psf, n_wavelets=K, levels=J) as p:
            p.set_schedule(ana_pipe=flip)
            p.op_analysis(dev(x, torch), u)
        assert rel_l2(host(u), ref) <= 1e-6
        got.append(u)
    assert torch.equal(*got)


def test_unaligned_coefficients():
    torch = cuda()
    import paper_1905_08468_gb300 as pkg
    lib = pkg.library()
    n, L, K, J = 256, 2, 4, 2
    x = np.random.default_rng(5).standard_normal((L, n, n)).astype(np.float32)
    xd = torch.empty(L * n * n + 1, device="cuda")
    xd[1:] = dev(x, torch).flatten()
    u = torch.full((L * K * n * n + 1,), float("nan"), device="cuda")
    st = lib.muffin_op_analysis_noalloc(ctypes.c_void_p(xd[1:].data_ptr()),
                                        ctypes.c_void_p(u[1:].data_ptr()), n, L, K, J,
                                        ctypes.c_void_p(torch.cuda.current_stream().cuda_stream))
    assert st == 0, lib.muffin_last_error().decode()
    torch.cuda.synchronize()
    ref = wavelets.Ws(x.astype(np.float64), daubechies.filter_bank(K), J)
    assert rel_l2(host(u[1:]).reshape(ref.shape), ref) <= 1e-6


@pytest.mark.parametrize("L,J", [(2, 1), (1, 3)])
def test_three_chains_masks(L, J):
    """Level 1 as the last level and above others with the derivatives' masks
    in a launch of their own."""
    from synth import make_cube
    from tests.test_gpu_states import run_case
    c = make_cube(128, L, 40, 2, 4000, seed=730 + J)
    run_case(c, (0.05, 0.05), 8, 3, (1e-5, 1e-4), levels=J)
