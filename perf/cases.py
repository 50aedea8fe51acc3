"""What is measured: the calls a program makes into the ISCI library, over the sizes it is used at.

Each case is one call (or one short call sequence) through the package's
public entry points on a context that the program has set up before: sigma
steps of full-CI, truncated and GAS spaces in both precisions, the batched
sigma of many instances, density matrices, propagation and the eigen-solver.
The integrals are the seeded synthetic sets of the benchmark and the tests
(synthetic.make_integrals, the paper's Be-in-a-box shape); CI vectors are
N(0, 1) vectors of unit norm.

exact() restates sigma, the density matrices, the propagation and the
eigenproblem in plain numpy / torch FP64 from the operators' definitions, with
its own strings, signs and screening.
"""
import itertools
import math

import numpy as np
import torch

from paper_1609_07757_gb300 import _lib as L
from paper_1609_07757_gb300.synthetic import make_integrals


def listed():
    return [
        # the smallest call: full CI of 2 + 2 electrons in 10 orbitals (the tests' size), launches and latency only
        dict(name="sigma_fci_n10", kind="sigma", n=10, na=2, nb=2, kmax=4, ell=3.0, nchol=20, box=False, tau=1e-14,
             nvec=1, precision=64),
        # the benchmark's workload: one FP64 sigma of full CI in 60 orbitals
        dict(name="sigma_fci_n60", kind="sigma", n=60, na=2, nb=2, kmax=4, ell=4.0, nchol=60, box=False, tau=1e-14,
             nvec=1, precision=64),
        # the largest full CI of the benchmark (24.5 M determinants)
        dict(name="sigma_fci_n100", kind="sigma", n=100, na=2, nb=2, kmax=4, ell=5.0, nchol=20, box=False, tau=1e-12,
             nvec=1, precision=64),
        # the FP32 form, as the mixed-precision solver calls it
        dict(name="sigma32_fci_n60", kind="sigma", n=60, na=2, nb=2, kmax=4, ell=4.0, nchol=60, box=False, tau=1e-14,
             nvec=1, precision=32),
        # more electrons in fewer orbitals: many hole strings, short contractions
        dict(name="sigma_fci_4a4b_n16", kind="sigma", n=16, na=4, nb=4, kmax=8, ell=3.0, nchol=20, box=False,
             tau=1e-14, nvec=1, precision=64),
        # the truncated spaces of the box sweep: triples, and singles and doubles (thin column classes)
        dict(name="sigma_cisdt_n100", kind="sigma", n=100, na=2, nb=2, kmax=3, ell=5.0, nchol=20, box=True, tau=1e-14,
             nvec=1, precision=64),
        dict(name="sigma_cisd_n100", kind="sigma", n=100, na=2, nb=2, kmax=2, ell=5.0, nchol=20, box=True, tau=1e-14,
             nvec=1, precision=64),
        # at most one electron in the continuum (GAS context), two vectors at once as a block solver hands them over
        dict(name="sigma_gas_n60_2vec", kind="gas", n=60, na=2, nb=2, ninner=20, ell=4.0, nchol=60, box=False,
             tau=1e-14, nvec=2, precision=64),
        # many independent instances of uneven size in one call
        dict(name="batch_sigma_16", kind="batch", count=16, lo=20, hi=60, na=2, nb=2, kmax=4, ell=3.0, nchol=20,
             box=False, tau=1e-14, nvec=1, precision=64),
        # one- and two-body density matrices of a state
        dict(name="density_fci_n60", kind="density", n=60, na=2, nb=2, kmax=4, ell=4.0, nchol=60, box=False, tau=1e-14,
             transition=False),
        # real-time steps under a field that couples through a one-body operator
        dict(name="propagate_fci_n41", kind="propagate", n=41, na=2, nb=2, kmax=4, ell=4.0, nchol=20, box=False,
             tau=1e-14, nsteps=2, krylov=14, dt=0.01),
        # the two lowest roots of a small space, start to finish (the solver's own kernels and host round trips)
        dict(name="davidson_fci_n10", kind="davidson", n=10, na=2, nb=2, kmax=4, ell=3.0, nchol=20, box=False,
             tau=1e-14, nroots=2, tol=1e-9),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more case of the ranges the listed ones stand for."""
    base = dict(na=2, nb=2, ell=rng.choice([3.0, 4.0, 5.0]), nchol=20, box=rng.random() < 0.3,
                tau=rng.choice([1e-14, 1e-12, 1e-10]))
    what = rng.choice(["fci", "fci", "fci", "wide", "trunc", "trunc", "fp32", "fp32", "gas", "batch", "density",
                       "propagate", "davidson"])
    nvec = rng.choice([1, 1, 2, 3])
    if what == "fci":
        n = _log_int(rng, 8, 96)
        if nvec > 1:
            n = min(n, 70)
        return dict(base, kind="sigma", n=n, kmax=4, nvec=nvec, precision=64)
    if what == "wide":
        na, nb, lo, hi = rng.choice([(3, 3, 9, 24), (4, 4, 9, 16), (3, 2, 9, 32), (4, 3, 9, 18)])
        return dict(base, kind="sigma", n=_log_int(rng, lo, hi), na=na, nb=nb, kmax=na + nb, nvec=1, precision=64)
    if what == "trunc":
        kmax = rng.choice([2, 3])
        return dict(base, kind="sigma", n=_log_int(rng, 20, 100), kmax=kmax, nvec=nvec, precision=64)
    if what == "fp32":
        return dict(base, kind="sigma", n=_log_int(rng, 20, 90), kmax=rng.choice([3, 4]), nvec=1, precision=32)
    if what == "gas":
        n = _log_int(rng, 20, 64)
        return dict(base, kind="gas", n=n, ninner=rng.randint(4, max(4, n // 2)), nvec=nvec, precision=64)
    if what == "batch":
        lo = rng.randint(12, 30)
        return dict(base, kind="batch", count=rng.randint(3, 16), lo=lo, hi=lo + rng.randint(5, 30), kmax=4, nvec=1,
                    precision=64)
    if what == "density":
        return dict(base, kind="density", n=_log_int(rng, 9, 56), kmax=rng.choice([2, 3, 4]),
                    transition=rng.random() < 0.5)
    if what == "propagate":
        return dict(base, kind="propagate", n=_log_int(rng, 9, 48), kmax=rng.choice([3, 4]), nsteps=rng.randint(1, 3),
                    krylov=rng.choice([12, 14, 16]), dt=0.01)
    return dict(base, kind="davidson", n=rng.randint(6, 10), kmax=4, nroots=rng.randint(1, 2), tol=1e-9)


# ---------------------------------------------------------------------------
# the program's side: contexts, vectors, calls


class _Context:
    """A library context that is destroyed with its owner."""

    def __init__(self):
        self.handle = L.iscsi_ctx_current()
        self.ndet = L.iscsi_ndet()

    def __del__(self):
        try:
            L.iscsi_ctx_destroy(self.handle)
        except Exception:  # the library may be gone at interpreter exit
            pass


def _gas_limits(case):
    """sizes, cmin, cmax of "at most one electron outside the inner orbitals"."""
    ne = case["na"] + case["nb"]
    return (case["ninner"], case["n"] - case["ninner"]), (ne - 1, ne), (ne, ne)


def _sizes(case, seed):
    """Orbital counts of the instances of a batch (the same for every seed: only the integrals change)."""
    rng = np.random.default_rng(case["count"] * 1000 + case["lo"])
    return [int(x) for x in rng.integers(case["lo"], case["hi"] + 1, size=case["count"])]


def _integrals(case, seed, n=None, instance=0):
    return make_integrals(n or case["n"], seed * 100 + instance, ell=case["ell"], nchol=case["nchol"],
                          box=case["box"])


def _vectors(seed, nvec, ndet):
    """N(0, 1) vectors of unit norm, FP64 on the GPU."""
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed)
    c = torch.randn(nvec, ndet, dtype=torch.float64, device="cuda", generator=gen)
    return c / c.norm(dim=1, keepdim=True)


def _phased(v, ref):
    """The program's phase convention: positive overlap with a fixed reference vector."""
    return v * torch.sign(v @ ref)[:, None]


def _coupling(n):
    """A dipole-like one-body operator: a position on the orbitals and its nearest-neighbour elements."""
    v = np.diag((np.arange(n) - (n - 1) / 2.0) / n)
    return v + 0.3 * (np.eye(n, k=1) + np.eye(n, k=-1))


def _field(case):
    return 0.05 * np.sin(0.8 * (np.arange(case["nsteps"]) + 0.5))


def _init(case, h1, eri):
    if case["kind"] == "gas":
        L.iscsi_init_gas(case["n"], case["na"], case["nb"], *_gas_limits(case), h1, eri, case["tau"])
    else:
        L.iscsi_init(len(h1), case["na"], case["nb"], case["kmax"], h1, eri, case["tau"])
    return _Context()


def prepare(case, seed):
    L.iscsi_set_stream(torch.cuda.current_stream())
    st = {"case": case}
    if case["kind"] == "batch":
        st["ctxs"] = [_init(case, *_integrals(case, seed, n, i)) for i, n in enumerate(_sizes(case, seed))]
        st["cs"] = [_vectors(seed * 100 + i, case["nvec"], x.ndet) for i, x in enumerate(st["ctxs"])]
        st["ss"] = [torch.empty_like(c) for c in st["cs"]]
        return st
    st["ctx"] = _init(case, *_integrals(case, seed))
    ndet = st["ctx"].ndet
    if case["kind"] in ("sigma", "gas"):
        st["c"] = _vectors(seed, case["nvec"], ndet)
        st["s"] = torch.empty_like(st["c"])
    elif case["kind"] == "density":
        n = case["n"]
        st["bra"] = _vectors(seed, 1, ndet)
        st["ket"] = _vectors(seed + 1, 1, ndet) if case["transition"] else None
        st["d1"] = torch.empty(2, n, n, dtype=torch.float64, device="cuda")
        st["d2"] = torch.empty(3, n, n, n, n, dtype=torch.float64, device="cuda")
    elif case["kind"] == "propagate":
        L.iscsi_init(case["n"], case["na"], case["nb"], case["kmax"], _coupling(case["n"]), None, case["tau"])
        st["cpl"] = _Context()
        st["c0"] = _vectors(seed, 2, ndet) / math.sqrt(2.0)
        st["c"] = torch.empty_like(st["c0"])
        st["field"] = _field(case)
    else:
        st["v"] = torch.empty(case["nroots"], ndet, dtype=torch.float64, device="cuda")
        st["ref"] = _vectors(0, 1, ndet)[0]
    return st


def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "batch":
        L.iscsi_batch_sigma([x.handle for x in state["ctxs"]], state["cs"], state["ss"], case["nvec"])
        return state["ss"]
    L.iscsi_ctx_use(state["ctx"].handle)
    if kind in ("sigma", "gas"):
        if case["precision"] == 32:
            L.iscsi_set_option("precision", 32)
            L.iscsi_sigma(state["c"], state["s"], case["nvec"])
            L.iscsi_set_option("precision", 64)
        else:
            L.iscsi_sigma(state["c"], state["s"], case["nvec"])
        return state["s"]
    if kind == "density":
        L.iscsi_density(state["bra"], state["ket"], state["d1"], state["d2"])
        return state["d1"], state["d2"]
    if kind == "propagate":
        state["c"].copy_(state["c0"])
        diag = L.iscsi_propagate(state["c"], case["nsteps"], case["dt"], state["field"], state["cpl"].handle,
                                 case["krylov"])
        return state["c"], diag[:, 1]
    status, energies = L.iscsi_davidson(case["nroots"], case["tol"], state["v"])
    if status != 0:
        raise RuntimeError("the eigen-solver did not converge")
    return energies, _phased(state["v"], state["ref"])


# ---------------------------------------------------------------------------
# work: updates of one sigma (one update = one sigma_I += unit * c_J over the
# determinant pairs of the space, every unit kept) and the arrays of the path


def _level_strings(n, ne, nocc):
    """Number of strings of each level (electrons outside the first nocc orbitals)."""
    return [math.comb(nocc, ne - l) * math.comb(n - nocc, l) if 0 <= ne - l <= nocc and l <= n - nocc else 0
            for l in range(ne + 1)]


def _steps(n, ne, nocc, l, k):
    """k-electron moves (k annihilated pairs' orbitals, k created) of a string of level l, by level change."""
    out = {}
    occ, vir = ne - l, l
    for i in range(k + 1):  # annihilated in the outer orbitals
        a = math.comb(vir, i) * math.comb(occ, k - i) if i <= vir and k - i <= occ else 0
        for j in range(k + 1):  # created in the outer orbitals
            fo, fv = nocc - (occ - (k - i)), (n - nocc) - (vir - i)
            b = math.comb(fv, j) * math.comb(fo, k - j) if 0 <= j <= fv and 0 <= k - j <= fo else 0
            if a * b:
                out[j - i] = out.get(j - i, 0) + a * b
    return out


def _space(case, n=None):
    """(n, na, nb, nocc_a, nocc_b, kmax) of the space the case's context works in."""
    n = n or case["n"]
    if case["kind"] == "gas":
        return n, case["na"], case["nb"], case["ninner"], case["ninner"], 1
    return n, case["na"], case["nb"], case["na"], case["nb"], case["kmax"]


def _counts(sp):
    """(determinants, updates of one sigma)."""
    n, na, nb, oa, ob, k = sp
    la, lb = _level_strings(n, na, oa), _level_strings(n, nb, ob)
    ndet = upd = 0
    for a, ca in enumerate(la):
        for b, cb in enumerate(lb):
            if a + b > k or not ca * cb:
                continue
            ndet += ca * cb
            a1, b1 = _steps(n, na, oa, a, 1), _steps(n, nb, ob, b, 1)
            per = sum(x * y for da, x in a1.items() for db, y in b1.items() if a + b + da + db <= k)
            for own in (a1, b1, _steps(n, na, oa, a, 2), _steps(n, nb, ob, b, 2)):
                per += sum(x for d, x in own.items() if a + b + d <= k)
            upd += per * ca * cb
    return ndet, upd


def work(case):
    if case["kind"] == "batch":
        got = [_counts(_space(case, n)) + (n,) for n in _sizes(case, 0)]
        return {"bytes": sum(16 * case["nvec"] * d + 2 * n**4 for d, _, n in got),
                "flops": sum(2 * case["nvec"] * u for _, u, _ in got)}
    n = case["n"]
    ndet, upd = _counts(_space(case))
    eri = 2 * n**4  # pair-packed integrals, 8 bytes each, the symmetric half
    if case["kind"] == "density":
        vecs = 2 if case["transition"] else 1
        return {"bytes": 8 * vecs * ndet + 8 * (2 * n**2 + 3 * n**4), "flops": 2 * upd}
    if case["kind"] == "propagate":
        sig = 2 * case["nsteps"] * case["krylov"]
        return {"bytes": 32 * ndet + eri, "flops": 2 * upd * sig}
    if case["kind"] == "davidson":
        return {"bytes": 8 * case["nroots"] * ndet + eri, "flops": 2 * upd * case["nroots"]}
    return {"bytes": 16 * case["nvec"] * ndet + eri, "flops": 2 * case["nvec"] * upd}


# ---------------------------------------------------------------------------
# exact: the same results in FP64 numpy / torch, from the operators themselves


def _dev(x, dtype=torch.float64):
    return torch.as_tensor(np.ascontiguousarray(x), device="cuda").to(dtype)


class _Spin:
    """Strings of one spin, sorted by (level, colex), with the one- and two-hole tables."""

    def __init__(self, n, ne, nocc):
        level = lambda s: sum(o >= nocc for o in s)  # noqa: E731
        self.n, self.ne = n, ne
        self.strings = sorted(itertools.combinations(range(n), ne), key=lambda s: (level(s), s[::-1]))
        self.level = np.array([level(s) for s in self.strings])
        at = {s: i for i, s in enumerate(self.strings)}
        self.count = len(self.strings)
        if ne >= 1:
            holes = list(itertools.combinations(range(n), ne - 1))
            hat = {s: i for i, s in enumerate(holes)}
            self.nx = len(holes)
            # a+_q |X>: string and sign (q, X); and per string its (X, q, sign)
            idx = np.full((n, self.nx), self.count)
            sgn = np.zeros((n, self.nx))
            dx = np.zeros((self.count, ne), dtype=np.int64)
            dq = np.zeros((self.count, ne), dtype=np.int64)
            ds = np.zeros((self.count, ne))
            for A, s in enumerate(self.strings):
                for i, q in enumerate(s):
                    x = hat[s[:i] + s[i + 1:]]
                    idx[q, x], sgn[q, x] = A, (-1.0) ** i
                    dx[A, i], dq[A, i], ds[A, i] = x, q, (-1.0) ** i
            self.idx, self.sgn = _dev(idx, torch.int64), _dev(sgn)
            self.dx, self.dq, self.ds = _dev(dx, torch.int64), _dev(dq, torch.int64), _dev(ds)
        if ne >= 2:
            pairs = list(itertools.combinations(range(n), 2))  # (low, high)
            pat = {p: i for i, p in enumerate(pairs)}
            holes = list(itertools.combinations(range(n), ne - 2))
            hat = {s: i for i, s in enumerate(holes)}
            self.pairs, self.nz = np.array(pairs), len(holes)
            idx = np.full((len(pairs), self.nz), self.count)
            sgn = np.zeros((len(pairs), self.nz))  # (-1)^(electrons of Z below low + below high)
            combos = list(itertools.combinations(range(ne), 2))
            dz = np.zeros((self.count, len(combos)), dtype=np.int64)
            dp, ds = dz.copy(), np.zeros((self.count, len(combos)))
            for A, s in enumerate(self.strings):
                for k, (i, j) in enumerate(combos):
                    z = hat[s[:i] + s[i + 1:j] + s[j + 1:]]
                    p = pat[(s[i], s[j])]
                    e = (-1.0) ** (i + j - 1)
                    idx[p, z], sgn[p, z] = A, e
                    dz[A, k], dp[A, k], ds[A, k] = z, p, e
            self.idx2, self.sgn2 = _dev(idx, torch.int64), _dev(sgn)
            self.dz, self.dp, self.ds2 = _dev(dz, torch.int64), _dev(dp, torch.int64), _dev(ds)


class _Exact:
    """H_tau on the full product of strings, cut to the space, in FP64."""

    def __init__(self, sp, tau, h1, eri):
        n, na, nb, oa, ob, kmax = sp
        self.n, self.tau = n, tau
        self.A, self.B = _Spin(n, na, oa), _Spin(n, nb, ob)
        keep = self.A.level[:, None] + self.B.level[None, :] <= kmax
        self.keep = torch.as_tensor(keep, device="cuda")
        self.shape = keep.shape
        h = np.where(np.abs(h1) > tau, h1, 0.0)
        self.h = _dev(h)
        self.G = None
        if eri is not None:
            i, j = np.meshgrid(np.arange(n), np.arange(n), indexing="ij")
            P = np.maximum(i, j) * (np.maximum(i, j) + 1) // 2 + np.minimum(i, j)
            P = torch.as_tensor(P.reshape(-1), device="cuda")
            g = _dev(eri)[P][:, P].reshape(n, n, n, n)  # (pq|rs)
            # same spin: a+_p a+_r a_q a_s with p > r, q > s carries g_psrq - g_pqrs; with the
            # pairs' signs kept apart (low, high) that is (g_pqrs - g_psrq) e_pr e_qs
            self.U = []
            for S in (self.A, self.B):
                if S.ne < 2:
                    self.U.append(None)
                    continue
                lo, hi = _dev(S.pairs[:, 0], torch.int64), _dev(S.pairs[:, 1], torch.int64)
                p, r, q, s = hi[:, None], lo[:, None], hi[None, :], lo[None, :]
                u = g[p, q, r, s] - g[p, s, r, q]
                self.U.append(torch.where(u.abs() > tau, u, torch.zeros_like(u)))
            g = torch.where(g.abs() > tau, g, torch.zeros_like(g))
            self.G = g.permute(0, 2, 1, 3).reshape(n * n, n * n).contiguous()  # rows (p, r), columns (q, s)
            del g

    def full(self, c):
        out = torch.zeros(self.shape, dtype=torch.float64, device="cuda")
        out[self.keep] = c
        return out

    def lift(self, C):
        """rows (q, s), columns (X, Y): s s C[X + q, Y + s]."""
        A, B, n = self.A, self.B, self.n
        Cp = torch.nn.functional.pad(C, (0, 1, 0, 1))
        x = Cp[A.idx.reshape(-1)][:, B.idx.reshape(-1)]
        x *= A.sgn.reshape(-1, 1)
        x *= B.sgn.reshape(1, -1)
        return x.reshape(n, A.nx, n, B.nx).permute(0, 2, 1, 3).reshape(n * n, A.nx * B.nx)

    def _one_spin(self, S, U, C):
        """One-body and same-spin parts for the spin whose strings are C's rows."""
        Cp = torch.nn.functional.pad(C, (0, 0, 0, 1))
        cols = C.shape[1]
        out = torch.zeros_like(C)
        if S.ne >= 1:
            x = Cp[S.idx.reshape(-1)] * S.sgn.reshape(-1, 1)
            t = (self.h @ x.reshape(self.n, S.nx * cols)).reshape(self.n, S.nx, cols)
            for i in range(S.ne):
                out += S.ds[:, i:i + 1] * t[S.dq[:, i], S.dx[:, i]]
        if U is not None:
            x = Cp[S.idx2.reshape(-1)] * S.sgn2.reshape(-1, 1)
            t = (U @ x.reshape(len(S.pairs), S.nz * cols)).reshape(len(S.pairs), S.nz, cols)
            for k in range(S.dz.shape[1]):
                out += S.ds2[:, k:k + 1] * t[S.dp[:, k], S.dz[:, k]]
        return out

    def sigma(self, c):
        A, B, n = self.A, self.B, self.n
        C = self.full(c)
        U = self.U if self.G is not None else (None, None)
        out = self._one_spin(A, U[0], C) + self._one_spin(B, U[1], C.T.contiguous()).T
        if self.G is not None and A.ne and B.ne:
            T = (self.G @ self.lift(C)).reshape(n, n, A.nx, B.nx)
            for i in range(A.ne):
                for j in range(B.ne):
                    out += (A.ds[:, i:i + 1] * B.ds[:, j][None, :]) * T[
                        A.dq[:, i][:, None], B.dq[:, j][None, :], A.dx[:, i][:, None], B.dx[:, j][None, :]]
        return out[self.keep]

    def density(self, bra, ket):
        n, A, B = self.n, self.A, self.B
        Cb, Ck = self.full(bra), self.full(ket)
        d1 = torch.zeros(2, n, n, dtype=torch.float64, device="cuda")
        d2 = torch.zeros(3, n, n, n, n, dtype=torch.float64, device="cuda")
        for s, (S, x, y) in enumerate(((A, Cb, Ck), (B, Cb.T.contiguous(), Ck.T.contiguous()))):
            xp, yp = (torch.nn.functional.pad(v, (0, 0, 0, 1)) for v in (x, y))
            if S.ne >= 1:
                lb, lk = ((v[S.idx.reshape(-1)] * S.sgn.reshape(-1, 1)).reshape(n, -1) for v in (xp, yp))
                d1[s] = lb @ lk.T
            if S.ne >= 2:
                lb, lk = ((v[S.idx2.reshape(-1)] * S.sgn2.reshape(-1, 1)).reshape(len(S.pairs), -1) for v in (xp, yp))
                q = lb @ lk.T
                lo, hi = _dev(S.pairs[:, 0], torch.int64), _dev(S.pairs[:, 1], torch.int64)
                e = torch.zeros(n * n, len(S.pairs), dtype=torch.float64, device="cuda")
                k = torch.arange(len(S.pairs), device="cuda")
                e[lo * n + hi, k], e[hi * n + lo, k] = 1.0, -1.0
                row = torch.zeros(n * n, dtype=torch.int64, device="cuda")
                row[lo * n + hi] = k
                row[hi * n + lo] = k
                sg = e.sum(1)
                full = q[row][:, row] * sg[:, None] * sg[None, :]  # (p, r), (q, t)
                d2[0 if s == 0 else 2] = full.reshape(n, n, n, n).permute(0, 2, 1, 3)
        if A.ne and B.ne:
            full = self.lift(Cb) @ self.lift(Ck).T
            d2[1] = full.reshape(n, n, n, n).permute(0, 2, 1, 3)
        return d1, d2

    def dense(self):
        nd = int(self.keep.sum())
        return torch.stack([self.sigma(e) for e in torch.eye(nd, dtype=torch.float64, device="cuda")], dim=1)


def _exact_of(case, seed, n=None, instance=0):
    return _Exact(_space(case, n), case["tau"], *_integrals(case, seed, n, instance))


def exact(case, seed):
    if case["kind"] == "batch":
        out = []
        for i, n in enumerate(_sizes(case, seed)):
            H = _exact_of(case, seed, n, i)
            c = _vectors(seed * 100 + i, case["nvec"], int(H.keep.sum()))
            out.append(torch.stack([H.sigma(v) for v in c]))
        return out
    H = _exact_of(case, seed)
    nd = int(H.keep.sum())
    if case["kind"] in ("sigma", "gas"):
        return torch.stack([H.sigma(v) for v in _vectors(seed, case["nvec"], nd)])
    if case["kind"] == "density":
        bra = _vectors(seed, 1, nd)[0]
        return H.density(bra, _vectors(seed + 1, 1, nd)[0] if case["transition"] else bra)
    if case["kind"] == "propagate":
        V = _Exact(_space(case), case["tau"], _coupling(case["n"]), None)
        c = _vectors(seed, 2, nd) / math.sqrt(2.0)
        energies = []
        for f in _field(case):
            Hc = lambda x: torch.stack([H.sigma(v) + f * V.sigma(v) for v in x])  # noqa: E731
            hx = Hc(c)
            energies.append(float((c * hx).sum() / (c * c).sum()))
            # the exponential's power series (|H| dt is a few at most)
            term, total, k = c, c.clone(), 0
            while float(term.norm()) > 1e-17:
                k += 1
                y = hx if k == 1 else Hc(term)
                term = torch.stack([y[1], -y[0]]) * (case["dt"] / k)
                total += term
            c = total
        return c, np.array(energies)
    w, v = torch.linalg.eigh(H.dense())
    return w[:case["nroots"]].cpu().numpy(), _phased(v[:, :case["nroots"]].T.contiguous(), _vectors(0, 1, nd)[0])
