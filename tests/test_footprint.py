"""A plan holds the spectral tables that its kernels read, and no others."""
import paper_1905_08468_gb300 as pkg


def test_no_dense_tables_where_the_fast_dct_runs():
    # 2 x 2 pixels, 1024 bands: everything but L x L tables (4 MiB each) is small
    for prec in ("tf32", "fp32"):
        assert pkg.estimate_bytes(2, 1024, n_wavelets=1, levels=1, precision=prec) < 4 << 20
    # a dense band count holds the folded tables (L x L values) only
    dense = pkg.estimate_bytes(2, 1000, n_wavelets=1, levels=1)
    fast = pkg.estimate_bytes(2, 1024, n_wavelets=1, levels=1)
    assert 0.9 * 4e6 < dense - fast < 1.1 * 4e6
