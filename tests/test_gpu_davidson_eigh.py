"""GPU: the solver's subspace eigen-decomposition against dense spectra.

Close and equal eigenvalues are where the refined FP32 rotations hand over to
FP64 ones; subspaces on both sides of the refinement's largest order.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from oracle import Oracle
from paper_1609_07757_gb300 import _lib as L
from paper_1609_07757_gb300.synthetic import make_integrals

pytestmark = pytest.mark.gpu


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


@pytest.mark.parametrize("gap", [0.0, 1e-13, 1e-9, 1e-5, 0.3])
@pytest.mark.parametrize("nroots", [1, 4, 7])
def test_close_roots(gap, nroots):
    """One-body levels in pairs `gap` apart, weak repulsion.  An energy with a residual r lies within |r|
    of a root (Weinstein), r below the solver's tolerance; inside a cluster narrower
    than that any mixture has converged."""
    n = 8
    lev = np.repeat([-2.0, -1.0, 0.5, 1.25], 2)
    lev[1::2] += gap
    q = np.linalg.qr(np.random.default_rng(11).standard_normal((n, n)))[0]
    h1 = (q * lev) @ q.T
    h1 = 0.5 * (h1 + h1.T)
    eri = 1e-3 * make_integrals(n, 3, ell=3.0, nchol=6)[1] if gap == 0.3 else np.zeros((n * (n + 1) // 2,) * 2)
    w = np.linalg.eigvalsh(Oracle(n, 2, 2, 4, 0.0, h1, eri).dense_h())
    L.iscsi_init(n, 2, 2, 4, h1, eri, 0.0)
    V = torch.zeros((nroots, L.iscsi_ndet()), dtype=torch.float64, device="cuda")
    st, e = L.iscsi_davidson(nroots, 1e-8, V)
    assert st == 0
    assert max(np.abs(w - x).min() for x in e) <= 1e-8
    assert abs(e[0] - w[0]) <= 1e-10
    G = (V @ V.T).cpu().numpy()
    assert np.abs(G - np.eye(nroots)).max() <= 1e-10
