"""What the tuner may read and store: choices that change a launch of the plan, timed on
the kernels of this library.  A choice without effect would be stored by noise
alone, and a line of a library whose choices meant other launches would pick
the wrong ones."""
import numpy as np
import pytest

from tests.gpu_util import cuda

pytestmark = pytest.mark.gpu


def plan(pkg, n, L, **kw):
    psf = np.zeros((L, n, n), np.float32)
    psf[:, 0, 0] = 1
    return pkg.Plan(n, L, psf, **kw)


@pytest.mark.parametrize("n,L,kw", [
    (16, 2, {}), (16, 4, {}), (32, 16, {}), (32, 128, {}), (64, 32, {}), (64, 128, {}),
    (32, 24, {}), (64, 8, {"precision": "fp32"}), (16, 16, {"dictionary": "iuwt"}),
    (32, 4, {"levels": 1}), (16, 8, {"sure": True, "levels": 2})])
def test_only_choices_with_an_effect_are_stored(tmp_path, n, L, kw):
    cuda()
    import paper_1905_08468_gb300 as pkg
    cache = tmp_path / "tune.txt"
    with plan(pkg, n, L, **kw) as p:
        assert p.autotune(str(cache)).from_cache == 0
    syn, ctas, tc, chunk, radix, order, ring, pipe = map(int, cache.read_text().split()[2:])
    if L & (L - 1) == 0:
        assert ctas == 0 and tc == 0                 # the fast DCT has no variants
    assert radix == 16 and ring == 0                 # one plan below 128 pixels a side
    if n in (32, 64):
        assert chunk == 0                            # the gradient is one kernel
    if kw.get("dictionary") == "iuwt":
        assert syn == 0 and pipe == 0
    if kw.get("levels") == 1:
        assert syn & 1 == 0                          # no coarse level
    if n < 64:
        assert pipe == 0                             # no level of the columns kernel
    if not kw.get("sure"):
        assert order == 0


def test_lines_of_earlier_kernels_are_not_used(tmp_path):
    cuda()
    import paper_1905_08468_gb300 as pkg
    cache = tmp_path / "tune.txt"
    with plan(pkg, 8, 5) as p:
        p.autotune(str(cache))
    key = cache.read_text().split()[1].replace("n=8,L=5", "n=8,L=6")
    old = ",".join(f for f in key.split(",") if not f.startswith("kernels="))
    cache.write_text("muffin-tune-6 %s 1 2 0 0 16 0 0 0\n" % old)
    with plan(pkg, 8, 6) as p:
        assert p.autotune(str(cache)).from_cache == 0
    key = key.replace("L=6", "L=7")
    cache.write_text("muffin-tune-6 %s 1 2 0 0 16 0 0 0\n" % key)
    with plan(pkg, 8, 7) as p:
        info = p.autotune(str(cache))
    assert info.from_cache == 1 and info.dct_ctas_per_sm == 2
