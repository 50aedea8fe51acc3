"""GPU: the contractions through residue numbers at the edges of their tiles and runs.

Reference: the FP64 FMA kernels of the same library (option fp64_tc = 0), which
share only the tables with the residue products.  Bars as in test_gpu_sigma
(1e-12 of the 2-norm and of the largest element): both routes round at about
1e-15 of the unit-weighted sums, whatever the sums' cancellation leaves of the
bar's three digits.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_1609_07757_gb300 import _lib as L
from paper_1609_07757_gb300.synthetic import make_integrals, transition_operator, unit_vector

pytestmark = pytest.mark.gpu

REL64 = 1e-12


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
    L.iscsi_set_option("fp64_tc", 1)
    L.iscsi_set_option("autotune", 1)


def sigma(C, nvec):
    c = torch.as_tensor(np.ascontiguousarray(C), dtype=torch.float64, device="cuda")
    s = torch.full_like(c, float("nan"))
    L.iscsi_sigma(c, s, nvec)
    torch.cuda.synchronize()
    return s.cpu().numpy()


def both(C, nvec):
    """sigma through residues (twice, bit for bit the same) and on the FMA kernels."""
    s = sigma(C, nvec)
    assert L.iscsi_stats()["residues"]["items"] > 0
    assert np.array_equal(s, sigma(C, nvec))
    L.iscsi_set_option("fp64_tc", 0)
    ref = sigma(C, nvec)
    L.iscsi_set_option("fp64_tc", 1)
    return s, ref


def check(s, ref):
    d = s - ref
    assert np.linalg.norm(d) <= REL64 * np.linalg.norm(ref)
    assert np.abs(d).max() <= REL64 * np.abs(ref).max()


# strings around 16, 64, 128 and 256 (tiles of C and M), pairs around 64 and 256 (K blocks and row
# tiles), one to five beta electrons (unrolled and general folds), unequal spins, runs of levels
SHAPES = [
    (7, 2, 2, 4), (11, 2, 2, 4), (12, 2, 2, 4), (16, 2, 2, 4), (17, 2, 2, 4), (23, 2, 2, 4), (24, 2, 2, 4),
    (20, 1, 1, 2), (12, 3, 3, 6), (9, 4, 4, 8), (11, 2, 5, 7), (11, 5, 2, 7), (13, 3, 1, 4),
    (17, 2, 2, 3), (24, 2, 2, 3), (12, 3, 3, 3), (12, 3, 3, 4), (10, 3, 4, 5),
]


@pytest.mark.parametrize("n,na,nb,kmax", SHAPES)
@pytest.mark.parametrize("nvec", [1, 3])
def test_residues_match_fma(n, na, nb, kmax, nvec):
    h1, eri = make_integrals(n, 7000 + n, ell=4.0, nchol=12)
    L.iscsi_init(n, na, nb, kmax, h1, eri, 1e-14)
    nd = L.iscsi_ndet()
    # vectors of different sizes: each has its own scale
    C = np.stack([unit_vector(nd, 10 + v) * 10.0 ** (3 * v) for v in range(nvec)])
    s, ref = both(C, nvec)
    for v in range(nvec):
        check(s[v], ref[v])


@pytest.mark.parametrize("what", ["constant", "graded", "single", "zero"])
def test_residues_extreme_vectors(what):
    # constant integrals and vector: every product of a chunk has the same sign and residues (the
    # largest sums); eight decades of magnitudes; one determinant; nothing
    n = 18
    h1, eri = make_integrals(n, 7100, ell=4.0, nchol=12)
    if what == "constant":
        h1, eri = np.ones_like(h1), np.ones_like(eri)
    L.iscsi_init(n, 2, 2, 4, h1, eri, 0.0)
    nd = L.iscsi_ndet()
    rng = np.random.default_rng(5)
    c = {"constant": np.full(nd, 1.0 / 3.0), "graded": rng.normal(size=nd) * 10.0 ** (-8 * rng.random(nd)),
         "single": np.eye(1, nd, nd // 3)[0], "zero": np.zeros(nd)}[what]
    s, ref = both(c[None], 1)
    if what == "zero":
        assert not s.any()
    else:
        check(s, ref)


# n, na, nb, kmax, transition: one tile, a tile and a remainder, classes that end inside a tile, one electron
# of a spin, K of less than one block and of several chunks
@pytest.mark.parametrize("n,na,nb,k,transition", [(16, 2, 2, 4, False), (17, 2, 2, 4, True), (19, 2, 2, 3, False),
                                                  (20, 2, 2, 2, True), (24, 2, 1, 3, False), (9, 4, 3, 7, True),
                                                  (8, 3, 3, 6, False)])
def test_density_residues(n, na, nb, k, transition):
    """Bar: 1e-12 of the block's largest element.  A coefficient's unit is 2^-57 of the vector's 2-norm and
    an element sums K products, so its error is below 2^-57 sqrt(K) of |bra| |ket| over the mean element,
    under 1e-14 of the largest one for these sizes."""
    h1, eri = make_integrals(n, 40 + n, ell=3.0, nchol=6)
    L.iscsi_init(n, na, nb, k, h1, eri, 0.0)
    nd = L.iscsi_ndet()
    bra = unit_vector(nd, 5) * 3e-150
    ket = unit_vector(nd, 6) * 7e120 if transition else bra
    bra[::7] *= 1e-9
    b = torch.as_tensor(bra, device="cuda")
    c = torch.as_tensor(ket, device="cuda") if transition else None
    d1 = torch.full((2, n, n), float("nan"), dtype=torch.float64, device="cuda")
    d2 = torch.full((3, n, n, n, n), float("nan"), dtype=torch.float64, device="cuda")
    L.iscsi_density(b, c, d1, d2)
    from oracle import Oracle
    r1, r2 = Oracle(n, na, nb, k, 0.0, h1, eri).density(bra, ket)
    for got, ref in [(d1.cpu().numpy(), np.asarray(r1))] + list(zip(d2.cpu().numpy(), np.asarray(r2))):
        assert np.abs(got - ref).max() <= 1e-12 * np.abs(ref).max()


# four strings' holes beyond the shared memory of half an SM: two holes per pass, without and with runs of levels
@pytest.mark.parametrize("kmax", [8, 5])
def test_residues_fold_in_passes(kmax):
    n = 15
    h1, eri = make_integrals(n, 7300, ell=4.0, nchol=12)
    L.iscsi_init(n, 4, 4, kmax, h1, eri, 1e-14)
    s, ref = both(unit_vector(L.iscsi_ndet(), 3)[None], 1)
    check(s[0], ref[0])


# more vectors than a thread block has threads, in both parts and in the string matrices' part alone (no
# two-electron part), single and in a batch; sizes over six decades, so that each vector's own exponent counts
@pytest.mark.parametrize("n,kmax,parts", [(10, 4, 3), (12, 4, 2)])
@pytest.mark.parametrize("batch", [False, True])
def test_residues_many_vectors(n, kmax, parts, batch):
    nvec = 300
    h1, eri = make_integrals(n, 7400, ell=3.0, nchol=12)
    L.iscsi_init(n, 2, 2, kmax, h1, eri if parts == 3 else None, 1e-14)
    nd = L.iscsi_ndet()
    C = np.stack([unit_vector(nd, 10 + v) * 10.0 ** (v % 7 - 3) for v in range(nvec)])
    s, ref = both(C, nvec)
    if batch:
        c = torch.as_tensor(C, device="cuda")
        out = torch.full_like(c, float("nan"))
        L.iscsi_batch_sigma([L.iscsi_ctx_current()], [c], [out], nvec)
        torch.cuda.synchronize()
        s = out.cpu().numpy()
    for v in range(nvec):
        check(s[v], ref[v])


def excitations(na, nb, kmax):
    """(number of differing alpha + beta orbitals of determinants i, j) as a function of i: a row over all j."""
    occ, lev = [], []
    for spin, ne in enumerate((na, nb)):
        o, l = L.iscsi_get_strings(spin, ne)
        m = np.zeros((len(l), 256), dtype=np.int64)
        m[np.arange(len(l))[:, None], np.asarray(o)] = 1
        occ.append(m)
        lev.append(np.asarray(l))
    A, B = np.nonzero(lev[0][:, None] + lev[1][None, :] <= kmax)  # determinants in order

    def row(i):
        same = (occ[0][A[i]] @ occ[0].T)[A] + (occ[1][B[i]] @ occ[1].T)[B]
        return occ[0][0].sum() + occ[1][0].sum() - same

    return row


# infinities and NaN: sigma is NaN exactly where H reaches them (within two excitations) and as without them
# elsewhere; more than the list holds: everywhere
@pytest.mark.parametrize("n,na,nb,kmax", [(18, 2, 2, 4), (24, 2, 2, 3), (9, 4, 4, 8), (12, 3, 3, 4), (20, 1, 1, 2),
                                          (11, 2, 5, 7)])
@pytest.mark.parametrize("count", [1, 3, 70])
def test_residues_nonfinite(n, na, nb, kmax, count):
    h1, eri = make_integrals(n, 7500 + n, ell=4.0, nchol=12)
    L.iscsi_init(n, na, nb, kmax, h1, eri, 1e-14)
    nd = L.iscsi_ndet()
    row = excitations(na, nb, kmax)
    rng = np.random.default_rng(n)
    at = rng.choice(nd, size=count, replace=False)
    bad = unit_vector(nd, 4)
    bad[at] = rng.choice([np.nan, np.inf, -np.inf], size=count)
    clean = np.where(np.isfinite(bad), bad, 0.0)
    # the second vector is finite, and the call after this one sees no trace of it
    s = sigma(np.stack([bad, clean]), 2)
    assert L.iscsi_stats()["residues"]["items"] > 0
    ref = sigma(clean[None], 1)[0]
    reached = np.any([row(i) <= 2 for i in at], axis=0) if count <= 64 else np.ones(nd, bool)
    assert np.isnan(s[0][reached]).all()
    for got in (s[0][~reached], s[1][~reached]):
        assert (np.abs(got - ref[~reached]) <= REL64 * np.abs(ref).max()).all()
    check(s[1], ref)


# coefficients that fall over 8 and 12 decades with the excitation level, and along the determinants
@pytest.mark.parametrize("n,na,nb,kmax", [(10, 2, 2, 4), (12, 2, 2, 3), (7, 3, 3, 6), (14, 2, 1, 3)])
@pytest.mark.parametrize("how,decades", [("level", 8), ("level", 12), ("index", 12)])
def test_residues_graded_elements(n, na, nb, kmax, how, decades):
    """Element by element.  A coefficient is rounded to 2^-58 of the largest one (half a unit of 2^(e - 58) with
    2^e <= 2 max|c|), a unit of H to 2^-50.9 of the largest opposite-spin one; so sigma_I is off by at most
    2^-58 max|c| sum_J |H_IJ| + 2^-50.9 g n_u sum_J |c_J| over the J that H reaches, with n_u the units that meet in
    an element of H (at most na nb + C(na, 2) + C(nb, 2) + na + nb), plus the reference's own rounding,
    2^-48 sum_J |H_IJ| |c_J| (columns of H from FP64 sums of up to 100 terms)."""
    h1, eri = make_integrals(n, 7600 + n, ell=3.0, nchol=20)
    L.iscsi_init(n, na, nb, kmax, h1, eri, 0.0)
    nd = L.iscsi_ndet()
    row = excitations(na, nb, kmax)
    rng = np.random.default_rng(7)
    fall = row(0) / (na + nb) if how == "level" else np.arange(nd) / nd
    c = rng.normal(size=nd) * 10.0 ** (-decades * fall)
    c /= np.linalg.norm(c)
    s = sigma(c[None], 1)[0]
    assert L.iscsi_stats()["residues"]["items"] > 0
    L.iscsi_set_option("fp64_tc", 0)
    H = np.concatenate([sigma(e, len(e)) for e in np.array_split(np.eye(nd), nd // 64 + 1)])  # symmetric
    L.iscsi_set_option("fp64_tc", 1)
    reach = np.stack([row(i) <= 2 for i in range(nd)])
    absH, absc = np.abs(H), np.abs(c)
    ref = (H.astype(np.longdouble) * c).sum(axis=1)
    units = na * nb + na * (na - 1) // 2 + nb * (nb - 1) // 2 + na + nb
    bar = (2.0 ** -58 * absc.max() * absH.sum(axis=1) + 2.0 ** -50.9 * np.abs(eri).max() * units * (reach @ absc)
           + 2.0 ** -48 * (absH @ absc))
    assert (np.abs(s - ref) <= bar).all()


def lifted_sizes(na, nb, kmax, c):
    """Per two-body block (aa, ab, bb): largest element and 1-norm of every row of the lifted vector, as matrices over
    the row's orbital pair."""
    occ, lev = [], []
    for spin, ne in enumerate((na, nb)):
        o, l = L.iscsi_get_strings(spin, ne)
        m = np.zeros((len(l), 64), dtype=bool)
        m[np.arange(len(l))[:, None], np.asarray(o)] = True
        occ.append(m)
        lev.append(np.asarray(l))
    C = np.zeros((len(lev[0]), len(lev[1])))
    C[lev[0][:, None] + lev[1][None, :] <= kmax] = np.abs(c)
    n = max(int(np.flatnonzero(o.any(0)).max()) for o in occ) + 1
    out = []
    for s, t in ((0, 0), (0, 1), (1, 1)):
        mx, one = np.zeros((n, n)), np.zeros((n, n))
        for p in range(n):
            for r in range(n):
                if s == t and p == r:
                    continue
                A = occ[0][:, p] & (occ[0][:, r] if t == 0 else True) if s == 0 else slice(None)
                B = occ[1][:, r] & (occ[1][:, p] if s == 1 else True) if t == 1 else slice(None)
                x = C[A][:, B]
                if x.size:
                    mx[p, r], one[p, r] = x.max(), x.sum()
        out.append((mx, one))
    return out


# coefficients that fall over 12 decades with the excitation level: element by element, ket = bra and a transition;
# long sums (14 moduli: 4 + 4 electrons), rows of a block split over several thread blocks
@pytest.mark.parametrize("n,na,nb,kmax,transition", [(8, 2, 2, 4, False), (9, 2, 2, 3, True), (7, 3, 2, 5, True),
                                                     (11, 3, 3, 6, False), (12, 4, 4, 8, True)])
def test_density_graded_elements(n, na, nb, kmax, transition):
    """A row's elements are integers of at least 50 bits below its largest one, so an element of d2 is off by at most
    2^-50 (max_x |L_y|_1 + max_y |L_x|_1); the reference's FP64 sums are within 2^-47 of the same bound (at most
    some thousand terms)."""
    h1, eri = make_integrals(n, 60 + n, ell=3.0, nchol=6)
    L.iscsi_init(n, na, nb, kmax, h1, eri, 0.0)
    nd = L.iscsi_ndet()
    fall = excitations(na, nb, kmax)(0) / (na + nb)
    vecs = [unit_vector(nd, 8 + i) * 10.0 ** (-12 * fall) for i in range(2 if transition else 1)]
    d1 = torch.full((2, n, n), float("nan"), dtype=torch.float64, device="cuda")
    d2 = torch.full((3, n, n, n, n), float("nan"), dtype=torch.float64, device="cuda")
    dev = [torch.as_tensor(v, device="cuda") for v in vecs]
    L.iscsi_density(dev[0], dev[1] if transition else None, d1, d2)
    from oracle import Oracle
    _, ref = Oracle(n, na, nb, kmax, 0.0, h1, eri).density(vecs[0], vecs[-1])
    ref = np.asarray(ref).reshape(3, n, n, n, n)
    sizes = [lifted_sizes(na, nb, kmax, v) for v in vecs]
    for got, want, (mx, ox), (my, oy) in zip(d2.cpu().numpy(), ref, sizes[0], sizes[-1]):
        # d2[p, q, r, t] = row (p, r) of bra times row (q, t) of ket
        bar = (2.0 ** -50 + 2.0 ** -47) * (mx[:, None, :, None] * oy[None, :, None, :]
                                           + my[None, :, None, :] * ox[:, None, :, None])
        assert (np.abs(got - want) <= bar).all()


@pytest.mark.parametrize("n,na,nb,kmax", [(8, 2, 2, 4), (9, 3, 2, 3)])
def test_density_nonfinite(n, na, nb, kmax):
    """A NaN makes the rows of the lifted vector that hold it NaN; the others are as without it."""
    h1, eri = make_integrals(n, 70 + n, ell=3.0, nchol=6)
    L.iscsi_init(n, na, nb, kmax, h1, eri, 0.0)
    nd = L.iscsi_ndet()
    bad = unit_vector(nd, 5)
    bad[nd // 2] = np.nan
    got = []
    for v in (bad, np.nan_to_num(bad, nan=0.0)):
        d2 = torch.zeros((3, n, n, n, n), dtype=torch.float64, device="cuda")
        L.iscsi_density(torch.as_tensor(v, device="cuda"), None, None, d2)
        got.append(d2.cpu().numpy())
    here = lifted_sizes(na, nb, kmax, (np.arange(nd) == nd // 2).astype(float))
    for blk, (a, b, (hit, _)) in enumerate(zip(*got, here)):
        reached = (hit[:, None, :, None] + hit[None, :, None, :]) > 0
        if blk != 1:  # elements with equal orbitals vanish by construction
            i = np.arange(n)
            reached[i, :, i, :] = reached[:, i, :, i] = False
        assert np.isnan(a[reached]).all() and np.array_equal(a[~reached], b[~reached])


# spaces on either side of each line of the routing: the same sigma whichever part takes the residues (3 both, 2 same
# spin, 1 opposite spin, 0 neither)
@pytest.mark.parametrize("n,na,nb,kmax,nvec", [(11, 3, 3, 4, 1), (11, 3, 3, 4, 12), (13, 4, 4, 4, 1), (10, 5, 4, 9, 1),
                                               (9, 4, 4, 8, 1), (12, 1, 4, 3, 4), (10, 5, 5, 3, 1), (14, 6, 1, 6, 2),
                                               (9, 1, 1, 2, 1), (18, 5, 1, 4, 1), (30, 3, 1, 2, 1),
                                               (13, 5, 1, 4, 1), (13, 1, 5, 4, 1), (13, 1, 5, 4, 2), (12, 5, 3, 4, 1),
                                               (19, 5, 1, 3, 1), (23, 1, 4, 5, 1), (11, 5, 5, 10, 1)])
def test_residues_routing(n, na, nb, kmax, nvec):
    h1, eri = make_integrals(n, 7700 + n, ell=3.0, nchol=12)
    L.iscsi_init(n, na, nb, kmax, h1, eri, 1e-14)
    C = np.stack([unit_vector(L.iscsi_ndet(), 30 + v) for v in range(nvec)])
    s = sigma(C, nvec)
    assert np.array_equal(s, sigma(C, nvec))
    L.iscsi_set_option("fp64_tc", 0)
    ref = sigma(C, nvec)
    for v in range(nvec):
        check(s[v], ref[v])


def test_autotune_leaves_no_slices_beside_residues():
    """The autotuner's other candidates cut the string matrices into slices; where the residues win, their memory is
    given back, a field step cuts nothing but residues, and the slices come back when they are asked for."""
    n = 40
    h1, eri = make_integrals(n, 7800, ell=4.0, nchol=12)
    L.iscsi_init(n, 2, 2, 4, h1, eri, 1e-14)
    c = unit_vector(L.iscsi_ndet(), 6)[None]
    L.iscsi_set_option("autotune", 1)
    s = sigma(c, 1)
    st = L.iscsi_stats()
    L.iscsi_set_option("autotune", 0)
    assert sum(t[3] >= 0 for t in st["route_fp64"]["trials"]) >= 2 and st["residues"]["items"] > 0
    assert st["samespin_slices"] == 0
    L.iscsi_set_option("fp64_tc", 0)
    check(s, sigma(c, 1))


def leave_free(nbytes):
    """Holds all of the device's memory but nbytes."""
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    return torch.empty(torch.cuda.mem_get_info()[0] - nbytes, dtype=torch.uint8, device="cuda")


def test_residues_make_room_for_another_context():
    """A context whose workspaces do not fit beside another one's residues (1.5 GB) gets their memory."""
    n = 60
    ints = [make_integrals(n, 7900 + i, ell=4.0, nchol=12) for i in range(2)]
    refs, hs = [], []
    for h1, eri in ints:
        L.iscsi_init(n, 2, 2, 4, h1, eri, 1e-14)
        c = unit_vector(L.iscsi_ndet(), 3)[None]
        L.iscsi_set_option("fp64_tc", 0)
        refs.append(sigma(c, 1))
        L.iscsi_set_option("fp64_tc", 1)
        L.iscsi_finalize()
    for h1, eri in ints:
        L.iscsi_init(n, 2, 2, 4, h1, eri, 1e-14)
        hs.append(L.iscsi_ctx_current())
    dev = torch.as_tensor(c, device="cuda")
    out = torch.empty_like(dev)
    L.iscsi_ctx_use(hs[0])
    L.iscsi_sigma(dev, out, 1)
    assert L.iscsi_stats()["residues"]["items"] > 0
    hog = leave_free(100 << 20)  # the second one's lifted vector and product take 208 MB
    try:
        got = []
        for h in (hs[1], hs[0]):
            L.iscsi_ctx_use(h)
            L.iscsi_sigma(dev, out, 1)
            got.append(out.cpu().numpy())
    finally:
        hog = None
        torch.cuda.empty_cache()
    check(got[0], refs[1])
    check(got[1], refs[0])


def test_residues_refused_for_a_large_block_only():
    """A block whose residues do not fit (40 vectors: 5 GB of 3.4 free) takes the slices; smaller ones take residues,
    before and after."""
    n, nvec = 40, 40
    h1, eri = make_integrals(n, 7950, ell=4.0, nchol=12)
    L.iscsi_init(n, 2, 2, 4, h1, eri, 1e-14)
    nd = L.iscsi_ndet()
    C = np.stack([unit_vector(nd, 50 + v) for v in range(nvec)])
    L.iscsi_set_option("fp64_tc", 0)
    ref = sigma(C, nvec)
    L.iscsi_finalize()
    L.iscsi_set_option("fp64_tc", 1)
    L.iscsi_init(n, 2, 2, 4, h1, eri, 1e-14)
    dev = torch.as_tensor(C, device="cuda")
    out = torch.empty_like(dev)
    hog = leave_free(5 << 30)
    try:
        items = []
        for k in (1, nvec, 1, nvec):
            out.fill_(float("nan"))
            L.iscsi_sigma(dev[:k], out[:k], k)
            items.append(L.iscsi_stats()["residues"]["items"])
            s = out.cpu().numpy()
            for v in range(k):
                check(s[v], ref[v])
    finally:
        hog = None
        torch.cuda.empty_cache()
    # (a block on the slices leaves the smaller one's residues where they are)
    assert items[0] > 0 and items[1] == 0 and items[2] == items[0]


# short sums over many rows
@pytest.mark.parametrize("n,na,nb,k,transition", [(26, 2, 1, 3, False), (30, 2, 1, 3, True), (27, 1, 1, 2, True),
                                                  (25, 1, 1, 2, False), (40, 2, 0, 2, False), (24, 1, 1, 2, True)])
def test_density_thin_blocks(n, na, nb, k, transition):
    h1, eri = make_integrals(n, 80 + n, ell=3.0, nchol=6)
    L.iscsi_init(n, na, nb, k, h1, eri, 0.0)
    nd = L.iscsi_ndet()
    bra = unit_vector(nd, 5)
    ket = unit_vector(nd, 6) if transition else bra
    d1 = torch.full((2, n, n), float("nan"), dtype=torch.float64, device="cuda")
    d2 = torch.full((3, n, n, n, n), float("nan"), dtype=torch.float64, device="cuda")
    b = torch.as_tensor(bra, device="cuda")
    L.iscsi_density(b, torch.as_tensor(ket, device="cuda") if transition else None, d1, d2)
    from oracle import Oracle
    r1, r2 = Oracle(n, na, nb, k, 0.0, h1, eri).density(bra, ket)
    for got, ref in [(d1.cpu().numpy(), np.asarray(r1))] + list(zip(d2.cpu().numpy(), np.asarray(r2))):
        assert np.abs(got - ref).max() <= 1e-12 * max(np.abs(ref).max(), 1e-300)


@pytest.mark.parametrize("kind", ["transition", "dense"])
def test_autotune_times_slices_for_one_body_operators(kind):
    """An operator without a two-body part: the slices skip the zero blocks of its string matrices, the residues do
    not, so both are timed; what the loser held is given back."""
    n = 60
    h1 = transition_operator(n, n - 1, 0) if kind == "transition" else make_integrals(n, 8100, ell=4.0, nchol=12)[0]
    L.iscsi_init(n, 2, 2, 4, h1, None, 0.0)
    c = unit_vector(L.iscsi_ndet(), 6)[None]
    L.iscsi_set_option("autotune", 1)
    s = sigma(c, 1)
    st = L.iscsi_stats()
    L.iscsi_set_option("autotune", 0)
    timed = {t[1]: t[3] for t in st["route_fp64"]["trials"] if t[0] == 1 and t[3] >= 0}
    assert 16 in timed and 64 in timed
    if timed[64] < min(t for k, t in timed.items() if k != 64):
        assert st["residues"]["items"] == 0 and st["samespin_slices"] == 1
    if timed[16] < min(t for k, t in timed.items() if k != 16):
        assert st["residues"]["items"] > 0 and st["samespin_slices"] == 0
    L.iscsi_set_option("fp64_tc", 0)
    check(s, sigma(c, 1))


@pytest.mark.parametrize("n,na,nb,kmax,nvec", [(17, 5, 1, 6, 1), (18, 4, 1, 3, 1), (19, 5, 1, 4, 1), (23, 1, 4, 5, 1),
                                               (35, 3, 1, 4, 1), (18, 4, 2, 4, 4), (14, 5, 2, 4, 1), (12, 4, 3, 4, 4)])
def test_residues_for_many_strings_and_electrons(n, na, nb, kmax, nvec):
    """Many strings of one spin or up to 15 pairs of electrons: both parts through residues, to their accuracy (the
    rounding of coefficients and integrals, 2^-58 and 2^-50 of the largest, at random in sums of K <= 5e3 terms of
    like size: below 1e-13 of the norm)."""
    h1, eri = make_integrals(n, 8200 + n, ell=3.0, nchol=12)
    L.iscsi_init(n, na, nb, kmax, h1, eri, 1e-14)
    C = np.stack([unit_vector(L.iscsi_ndet(), 30 + v) for v in range(nvec)])
    s = sigma(C, nvec)
    assert L.iscsi_stats()["residues"]["items"] > 0
    L.iscsi_set_option("fp64_tc", 0)
    ref = sigma(C, nvec)
    for v in range(nvec):
        assert np.linalg.norm(s[v] - ref[v]) <= 1e-13 * np.linalg.norm(ref[v])
