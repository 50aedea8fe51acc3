"""GPU: the FP32 form at both tile widths, stages and chunks that end inside one another.

Reference: the FP64 sigma of the same library.  Bar: 5e-6 of the 2-norm (products
to 2^-24, FP32 sums of some thousand terms).
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_1609_07757_gb300 import _lib as L
from paper_1609_07757_gb300.synthetic import make_integrals, unit_vector

pytestmark = pytest.mark.gpu

REL32 = 5e-6


@pytest.fixture(autouse=True)
def _fresh_library():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    L.load()
    L.iscsi_set_option("autotune", 0)
    L.iscsi_set_stream(torch.cuda.current_stream())
    yield
    torch.cuda.synchronize()
    L.iscsi_finalize()
    L.iscsi_set_option("autotune", 1)


# full CI: one narrow wave, wide tiles (the same-spin part's 49 + 49 K steps: half stages, chunks ending inside
# a stage), two vectors; truncated: segments of unequal reach (narrow at any size)
@pytest.mark.parametrize("n,na,nb,k,nvec", [(20, 2, 2, 4, 1), (40, 2, 2, 4, 1), (43, 2, 2, 4, 2), (40, 2, 1, 3, 1),
                                            (46, 2, 2, 3, 1), (60, 2, 2, 2, 2)])
def test_fp32_form_against_fp64(n, na, nb, k, nvec):
    h1, eri = make_integrals(n, 60 + n, ell=4.0, nchol=8)
    L.iscsi_init(n, na, nb, k, h1, eri, 1e-14)
    nd = L.iscsi_ndet()
    c = torch.as_tensor(np.stack([unit_vector(nd, 7 + v) for v in range(nvec)]), device="cuda")
    out = {}
    for prec in (64, 32):
        L.iscsi_set_option("precision", prec)
        s = torch.full_like(c, float("nan"))
        L.iscsi_sigma(c, s, nvec)
        torch.cuda.synchronize()
        out[prec] = s.cpu().numpy()
    L.iscsi_set_option("precision", 64)
    for v in range(nvec):
        assert np.linalg.norm(out[32][v] - out[64][v]) <= REL32 * np.linalg.norm(out[64][v])


@pytest.mark.parametrize("n,na,nb,k", [(24, 2, 2, 4), (22, 3, 2, 5), (44, 2, 2, 3)])
def test_fp32_form_bits_do_not_depend_on_the_tiles(n, na, nb, k):
    # one vector fills a wave of narrow tiles at most, a block of sixteen many: the launch takes another tile width and
    # other tiles, and every vector comes out with the same bits
    h1, eri = make_integrals(n, 90 + n, ell=4.0, nchol=8)
    L.iscsi_init(n, na, nb, k, h1, eri, 1e-14)
    c = torch.as_tensor(np.stack([unit_vector(L.iscsi_ndet(), 7 + v) for v in range(16)]), device="cuda")
    L.iscsi_set_option("precision", 32)
    try:
        block = torch.empty_like(c)
        L.iscsi_sigma(c, block, 16)
        one = torch.empty_like(c[:1])
        for v in (0, 5, 15):
            L.iscsi_sigma(c[v:v + 1], one, 1)
            assert torch.equal(one[0], block[v])
    finally:
        L.iscsi_set_option("precision", 64)
