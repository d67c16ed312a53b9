"""FP64 products from digits, entry by entry (csrc/oz_gemm.cu).

Basis functions, points and orbitals sit on a line and decay with the distance,
so that the large entries of most operand rows meet small ones of the other
row: sum |a||b| falls to 10^-decay of the product of the two largest, and
digits relative to those largest are not enough.

Bound: every product, from its own operands as the library holds them, to
(4 K + 2) u sum_k |a_k||b_k| of each entry (u = 2^-53).  An FP64 loop over K
complex terms has 2 K u; digits that are kept where S = sum |a||b| 2^-(ea+eb) is
at least 2^-10 err by at most 2 K 2^-62 = K u 2^-8 of 2^(ea+eb) before the final
rounding, so 4 K u sum |a||b|.  The references are sums in 64-bit mantissas or
better (error 2 K 2^-64, inside the slack of the bound)."""
import numpy as np
import pytest

from oracle import setup_oracle as S
from paper_2304_05505_gb300 import cells

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

U = 2.0 ** -53


@pytest.fixture(scope="module")
def thc(cuda_required):
    import os

    from paper_2304_05505_gb300 import build_lib, thc as mod
    if not os.path.exists(mod.LIB_PATH):
        build_lib.build()
    mod.load()
    yield mod
    mod.thc_debug_limit_scratch(-1)


def _two_prod(a, b):
    """a b = p + e exactly (Dekker)."""
    p = a * b
    c = 134217729.0
    ah = a * c - (a * c - a)
    bh = b * c - (b * c - b)
    al, bl = a - ah, b - bh
    return p, ((ah * bh - p) + ah * bl + al * bh) + al * bl


def _sum2(re, p):
    """re + p in a float-float pair."""
    hi, lo = re
    s = hi + p
    bb = s - hi
    return s, lo + ((hi - (s - bb)) + (p - bb))


def _product_errors(A, B, C):
    """|C - A B^T| over sum |a||b| per entry, A [m, K], B [n, K] complex, in doubled precision."""
    m, K = A.shape
    n = B.shape[0]
    re, im = (np.zeros((m, n)), np.zeros((m, n))), (np.zeros((m, n)), np.zeros((m, n)))
    for k in range(K):
        ar, ai = A[:, k].real[:, None], A[:, k].imag[:, None]
        br, bi = B[:, k].real[None, :], B[:, k].imag[None, :]
        for x, y, acc, sign in ((ar, br, 0, 1), (ai, bi, 0, -1), (ar, bi, 1, 1), (ai, br, 1, 1)):
            p, e = _two_prod(x, y)
            if acc == 0:
                re = _sum2(re, sign * p)
                re = (re[0], re[1] + sign * e)
            else:
                im = _sum2(im, sign * p)
                im = (im[0], im[1] + sign * e)
    den = np.abs(A) @ np.abs(B).T
    er = np.abs((re[0] - C.real) + re[1])
    ei = np.abs((im[0] - C.imag) + im[1])
    return np.maximum(er, ei) / den


def _line(rng, shape, x, y, decay):
    a = rng.normal(size=shape) + 1j * rng.normal(size=shape)
    return a * 10.0 ** (-decay * np.abs(x[:, None] - y[None, :]))


@pytest.mark.parametrize("decay", [4.0, 14.0, 60.0])
@pytest.mark.parametrize("mesh,nbas,nocc,nisdf", [
    ((2, 1, 1), 130, 70, 301),
    ((1, 1, 1), 96, 41, 410),
])
def test_build_products_entry_by_entry(thc, mesh, nbas, nocc, nisdf, decay):
    rng = np.random.default_rng(int(decay) + nisdf)
    nk = int(np.prod(mesh))
    xm, xp, xi = (np.sort(rng.uniform(size=n)) for n in (nbas, nisdf, nocc))
    X = _line(rng, (nk, nbas, nisdf), xm, xp, decay)
    C = _line(rng, (nk, nbas, nocc), xm, xi, decay)
    V = cells.random_problem(mesh, nbas=8, nocc=3, nisdf=nisdf, seed=3)["V"]
    eb = thc.ExchangeBuild(dict(n1=mesh[0], n2=mesh[1], n3=mesh[2], nbas=nbas, nocc=nocc, nisdf=nisdf), "fp64")
    try:
        eb.set_collocation(X)
        eb.set_kernel(V)
        KC, _ = eb.build(C)
        eb.sync()
        KC = KC.cpu().numpy()
        Psi, D, M, Y = (eb.intermediate(i).cpu().numpy() for i in range(4))
    finally:
        eb.close()
    for k in range(nk):
        for what, A, B, R in (("S1", X[k].T, C[k].T, Psi[k]), ("S2", Psi[k], Psi[k].conj(), D[k]),
                              ("S4a", M[k], Psi[k].T, Y[k]), ("S4b", X[k].conj(), Y[k].T, KC[k])):
            err = _product_errors(A, B, R).max()
            assert err <= (4 * A.shape[1] + 2) * U, (what, err)


@pytest.mark.parametrize("nbas", [33, 432, 1500])
def test_many_small_entries_beside_a_large_one(thc, nbas):
    """Rows of X^T with one large entry, where C is zero, and small ones, so
    that S = sum |a||b| 2^-(ea+eb) is 2^-10 to 2^-4: it falls only as far as the
    small entries do, and each of their roundings counts.

    Bound: 6 u sum |a||b| (u = 2^-53).  Digits are kept where their roundings'
    rms is at most 2^-53.3 sum |a||b| = 0.81 u; 6 sigma over 2^17 entries and
    the final rounding make 5.4 u.  FP64 sums of random signs leave u
    sum |a||b| times about 0.5 rms, 3 u at 6 sigma."""
    rng = np.random.default_rng(nbas)
    nocc, nisdf = 31, 260
    X = rng.normal(size=(1, nbas, nisdf)) + 1j * rng.normal(size=(1, nbas, nisdf))
    # (C's columns have entries of about 0.28 of their scale, so S = 0.31 nbas 2^-s)
    X *= 2.0 ** -(np.log2(0.31 * nbas) + rng.uniform(4, 9.8, size=(1, 1, nisdf)))
    X[0, 0] = 0.9
    C = rng.normal(size=(1, nbas, nocc)) + 1j * rng.normal(size=(1, nbas, nocc))
    C[0, 0] = 0.0
    eb = thc.ExchangeBuild(dict(n1=1, n2=1, n3=1, nbas=nbas, nocc=nocc, nisdf=nisdf), "fp64")
    try:
        eb.set_collocation(X)
        eb.set_kernel(cells.random_problem((1, 1, 1), nbas=8, nocc=3, nisdf=nisdf, seed=3)["V"])
        eb.build(C)
        eb.sync()
        Psi = eb.intermediate(0).cpu().numpy()
    finally:
        eb.close()
    assert _product_errors(X[0].T, C[0].T, Psi[0]).max() <= 6 * U


@pytest.mark.parametrize("where", ["inf", "nan", "both"])
def test_nonfinite_coefficients_spread_as_in_fp64_sums(thc, where):
    """An Inf or a NaN in C reaches the entries that it reaches on the FP64
    pipe (the call without scratch), and as the same kind of number."""
    r = cells.random_problem((1, 1, 1), nbas=90, nocc=70, nisdf=301, seed=5)
    C = np.array(r["C"])
    if where != "nan":
        C[0, 3, 7] = complex(np.inf, 0.5)
    if where != "inf":
        C[0, 60, 33] = complex(0.25, np.nan)
    eb = thc.ExchangeBuild(dict(n1=1, n2=1, n3=1, nbas=90, nocc=70, nisdf=301), "fp64")
    try:
        eb.set_collocation(r["X"])
        eb.set_kernel(r["V"])
        got = []
        for limit in (-1, 0):
            thc.thc_debug_limit_scratch(limit)
            eb.build(C)
            eb.sync()
            got.append([eb.intermediate(i).cpu().numpy().view(np.float64) for i in (0, 1)])
    finally:
        thc.thc_debug_limit_scratch(-1)
        eb.close()
    for a, b in zip(*got):
        assert not np.isfinite(a).all()
        assert np.array_equal(np.isnan(a), np.isnan(b))
        assert np.array_equal(np.where(np.isinf(a), np.sign(a), 0), np.where(np.isinf(b), np.sign(b), 0))


@pytest.mark.parametrize("decay", [2.0, 6.0, 14.0])
def test_selection_on_localised_orbitals(thc, decay):
    """Blocks of pivots on orbitals that decay along a line: the oracle's
    points, and residuals to 1e-10 of each candidate's own diagonal entry
    (60 rows of sums of 210 terms, divided by pivots above 1e-4 of their
    diagonal: 1e4 x 270 x 2^-53 = 3e-10 at the worst, a third of it allowed)."""
    rng = np.random.default_rng(int(decay))
    nf, nr, npts = 210, 5200, 60
    Uo = _line(rng, (nf, nr), np.sort(rng.uniform(size=nf)), np.sort(rng.uniform(size=nr)), decay)
    Uo = Uo * np.exp(0.5 * rng.normal(size=(1, nr)))
    ref = S.pivoted_cholesky(Uo, npts)
    pts, resid = thc.thc_select_points(torch.from_numpy(Uo).cuda(), npts)
    assert np.array_equal(pts, ref["points"])
    own = (np.abs(Uo) ** 2).sum(0) ** 2
    assert (np.abs(resid.cpu().numpy() - ref["resid"]) <= 1e-10 * own).all()


@pytest.mark.parametrize("mesh", [(4, 4, 4), (3, 3, 3), (2, 4, 1), (1, 3, 2), (1, 1, 1)])
def test_nonfinite_elements_of_the_convolution(thc, mesh):
    """A NaN, an Inf or a product that overflows in the fixed-point convolution
    leaves its element what the general FP64 transform makes of it, butterfly by
    butterfly (numpy below), and touches no other element."""
    nk, npq = int(np.prod(mesh)), 70
    rng = np.random.default_rng(nk)
    D = rng.normal(size=(nk, npq)) + 1j * rng.normal(size=(nk, npq))
    V = rng.normal(size=(nk, npq)) + 1j * rng.normal(size=(nk, npq))
    D[nk - 1, 5] = complex(np.inf, 0.0)
    D[0, 11] = complex(0.5, np.nan)
    D[:, 23] = complex(1e200, 0.0) * rng.normal(size=nk)
    V[:, 23] = complex(1e200, 0.0) * rng.normal(size=nk)
    D[0, 64] = complex(-np.inf, 0.0)
    D[1 % nk, 64] = complex(np.inf, 1.0)

    def axis(x, sign):       # along the first axis, the butterflies of the library
        n = x.shape[0]
        i = lambda z: np.stack([-sign * z[..., 1], sign * z[..., 0]], -1)
        if n == 2:
            return np.stack([x[0] + x[1], x[0] - x[1]])
        if n == 3:
            t, d = x[1] + x[2], x[1] - x[2]
            m, s = x[0] - 0.5 * t, i(0.86602540378443864676 * d)
            return np.stack([x[0] + t, m + s, m - s])
        if n == 4:
            a0, a1, b0, b1 = x[0] + x[2], x[0] - x[2], x[1] + x[3], i(x[1] - x[3])
            return np.stack([a0 + b0, a1 + b1, a0 - b0, a1 - b1])
        return x

    def dft(x, sign):
        x = x.reshape(mesh + (npq, 2))
        for a in range(3):
            x = np.moveaxis(axis(np.moveaxis(x, a, 0), sign), 0, a)
        return x.reshape(nk, npq, 2)

    def cmul(a, b):
        return np.stack([a[..., 0] * b[..., 0] - a[..., 1] * b[..., 1], a[..., 0] * b[..., 1] + a[..., 1] * b[..., 0]], -1)

    with np.errstate(all="ignore"):
        pair = lambda z: np.stack([z.real, z.imag], -1)
        vh = dft(pair(V), +1) / nk
        ref = dft(cmul(dft(pair(D), -1), vh), +1)
    M = torch.empty((nk, npq), dtype=torch.complex128, device="cuda")
    thc.thc_kconv_noalloc(torch.from_numpy(D).cuda(), torch.from_numpy(V).cuda(), M, mesh, npq)
    got = pair(M.cpu().numpy())
    assert np.array_equal(np.isnan(got), np.isnan(ref))
    assert np.array_equal(np.where(np.isinf(got), np.sign(got), 0), np.where(np.isinf(ref), np.sign(ref), 0))
    fine = np.isfinite(ref).all(axis=(0, 2))
    assert set(np.nonzero(~fine)[0]) <= {5, 11, 23, 64}
    scale = np.abs(ref).max(axis=(0, 2), where=np.isfinite(ref), initial=0)
    assert (np.abs(got[:, fine] - ref[:, fine]) <= 1e-14 * nk * scale[None, fine, None]).all()
