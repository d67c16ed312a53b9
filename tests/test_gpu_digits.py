"""FP64 products on the tensor cores (csrc/oz_gemm.cu) and the blocked Cholesky
inverse (csrc/chol.cu) at the sizes where they can go wrong, through the fit.

The orbitals are unstructured (complex Gaussian), so the metric S = |B|^2 of
the points is well conditioned (below 1e3 for these sizes) and xi, V follow
the FP64 oracle to about cond(S) * 1e-16 * sqrt(K); the bound is 1e-12 of the
largest entry.  The shapes cross the edges of the 128 x 80 output tile, the
32-deep stage and the 64-deep exact chunk (real K = 2 * orbitals), the
32-column panels of the factor and the 256-row level of its inverse that runs
on the tensor cores."""
import numpy as np
import pytest

from oracle import setup_oracle as S

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def thc(cuda_required):
    import os

    from paper_2304_05505_gb300 import build_lib, thc as mod
    if not os.path.exists(mod.LIB_PATH):
        build_lib.build()
    mod.load()
    return mod


@pytest.mark.parametrize("nfunc,grid,npts", [
    (16, (7, 9, 5), 31),      # one stage of K, one panel
    (17, (16, 12, 11), 33),   # a stage and a remainder, two panels
    (32, (10, 13, 17), 40),   # the columns of one tile exactly (40 points embedded)
    (33, (16, 16, 16), 41),   # a chunk and a remainder, one column past a tile
    (70, (12, 11, 13), 129),
    (90, (15, 16, 17), 300),  # the inverse's level of 256 rows
    (60, (13, 14, 15), 520),
])
def test_fit_on_unstructured_orbitals(thc, nfunc, grid, npts):
    rng = np.random.default_rng(nfunc)
    ng = int(np.prod(grid))
    U = rng.normal(size=(nfunc, ng)) + 1j * rng.normal(size=(nfunc, ng))
    U *= np.exp(rng.normal(size=(nfunc, 1)))            # rows of different size
    lat = np.diag([5.0, 6.0, 7.0])
    pts = np.sort(rng.permutation(ng)[:npts])
    V, xi = thc.thc_fit_kernel(torch.from_numpy(U).cuda(), grid, lat, (1, 1, 2), pts, want_xi=True)
    ref = S.fit_kernel(lat, grid, (1, 1, 2), U, pts)
    xr = S.isdf_fit(U, pts)
    assert np.abs(xi.cpu().numpy() - xr).max() <= 1e-12 * np.abs(xr).max()
    assert np.abs(V.cpu().numpy() - ref).max() <= 1e-12 * np.abs(ref).max()


def test_fit_of_nonfinite_orbitals_is_rejected(thc):
    """A NaN in an orbital reaches the metric, whose pivots then fail."""
    U = torch.randn(24, 13 * 14 * 15, dtype=torch.complex128, device="cuda")
    U[3, 5] = complex("nan")
    with pytest.raises(thc.ThcError):
        thc.thc_fit_kernel(U, (13, 14, 15), np.diag([5.0, 5.0, 5.0]), (1, 1, 1), np.arange(40))


@pytest.mark.parametrize("mesh,nbas,nocc,nisdf", [
    ((4, 4, 4), 33, 20, 79),     # radix-4 lanes; N_P one short of a tile's columns
    ((3, 3, 3), 40, 33, 129),    # radix-3 lanes
    ((2, 4, 3), 65, 16, 81),     # mixed axes
    ((1, 3, 2), 96, 64, 256),    # one lane an element, whole tiles
    ((4, 1, 1), 130, 41, 333),
])
def test_fp64_build_from_digits(thc, mesh, nbas, nocc, nisdf):
    """The FP64 build whose products and k-convolution run from digits and in
    fixed point, against the FP64 oracle: each step rounds once at 2^-53 of
    its result (the sums are exact to 2^-60), so the bound is 1e-13 of the
    largest entry, of E_x and of the Hermitian deviation."""
    from oracle import thc_oracle as O
    from paper_2304_05505_gb300 import cells
    r = cells.random_problem(mesh, nbas=nbas, nocc=nocc, nisdf=nisdf, seed=nisdf)
    ref = O.build(r["X"], r["C"], r["V"], r["mesh"], route="direct", keep=True)
    eb = thc.ExchangeBuild(dict(n1=mesh[0], n2=mesh[1], n3=mesh[2], nbas=nbas, nocc=nocc, nisdf=nisdf), "fp64")
    eb.set_collocation(r["X"])
    eb.set_kernel(r["V"])
    KC, ex = eb.build(r["C"])
    eb.sync()
    assert np.abs(KC.cpu().numpy() - ref["KC"]).max() <= 1e-13 * np.abs(ref["KC"]).max()
    assert abs(float(ex[0]) - ref["Ex"]) <= 1e-13 * abs(ref["Ex"])
    K, ex2 = eb.build_K(r["C"])
    eb.sync()
    Kr = np.einsum("kmp,kpq,knq->kmn", r["X"].conj(), ref["M"], r["X"])
    assert np.abs(K.cpu().numpy() - Kr).max() <= 1e-13 * np.abs(Kr).max()
    eb.close()


@pytest.mark.parametrize("mesh", [(4, 4, 4), (3, 2, 1)])
def test_fixed_point_convolution_range(thc, mesh):
    """The k-convolution of values spread over 40 orders of magnitude between
    the elements (each has its own scale), and of a NaN, which reaches every
    k of its own element and no other."""
    nk, npq = int(np.prod(mesh)), 50
    rng = np.random.default_rng(3)
    s = 10.0 ** rng.uniform(-20, 20, size=npq)
    D = (rng.normal(size=(nk, npq)) + 1j * rng.normal(size=(nk, npq))) * s
    V = (rng.normal(size=(nk, npq)) + 1j * rng.normal(size=(nk, npq))) / s ** 2
    d = np.fft.fftn(D.reshape(mesh + (npq,)), axes=(0, 1, 2))
    v = np.fft.ifftn(V.reshape(mesh + (npq,)), axes=(0, 1, 2)) * nk
    ref = np.fft.ifftn(d * v, axes=(0, 1, 2)).reshape(nk, npq)
    D[nk - 1, 7] = complex(0.0, float("nan"))
    M = torch.empty((nk, npq), dtype=torch.complex128, device="cuda")
    thc.thc_kconv_noalloc(torch.from_numpy(D).cuda(), torch.from_numpy(V).cuda(), M, mesh, npq)
    got = M.cpu().numpy()
    assert np.isnan(got[:, 7]).all()
    keep = np.arange(npq) != 7
    assert (np.abs(got - ref)[:, keep] <= 1e-14 * np.abs(ref).max(0)[keep]).all()


def _pair_orbitals(kind, nf, nr, seed):
    rng = np.random.default_rng(seed)
    U = rng.normal(size=(nf, nr)) + 1j * rng.normal(size=(nf, nr))
    if kind == "spread":         # residuals over several orders: few candidates per bin
        U *= np.exp(0.5 * rng.normal(size=(1, nr)))
    elif kind == "rank":         # pair Gram of rank 25: the trace ends the selection inside a block
        U = rng.normal(size=(nf, 5)) @ (U[:5] * np.exp(0.3 * rng.normal(size=(1, nr))))
    elif kind == "flat":         # more than 800 candidates within a bin of the largest: single pivots
        U *= (1 + 1e-4 * rng.uniform(size=nr)) / np.sqrt((np.abs(U) ** 2).sum(0))
    return U


@pytest.mark.parametrize("kind,nf,nr,npts", [
    ("spread", 700, 1600, 20),      # the smallest selection that goes in blocks
    ("spread", 450, 2305, 41),      # a block and one pivot
    ("spread", 410, 2500, 130),     # earlier rows' products in the later blocks
    ("rank", 420, 2400, 64),
    ("flat", 420, 2400, 24),
])
def test_pivots_in_blocks_match_oracle(thc, kind, nf, nr, npts):
    """Selections large enough to go in blocks of pivots take the oracle's
    points in its order, and leave its residuals to 1e-12 of the largest
    diagonal entry (sums of at most 130 rows, each rounded once)."""
    U = _pair_orbitals(kind, nf, nr, npts)
    ref = S.pivoted_cholesky(U, npts)
    pts, resid = thc.thc_select_points(torch.from_numpy(U).cuda(), npts)
    assert np.array_equal(pts, ref["points"])
    scale = float((np.sum(np.abs(U) ** 2, axis=0) ** 2).max())
    assert np.abs(resid.cpu().numpy() - ref["resid"]).max() <= 1e-12 * scale
