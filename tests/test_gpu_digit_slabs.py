"""Digit products that do not fit their scratch whole (csrc/oz_gemm.cu): taken
in slabs of the batch, of lane rows and of column rows they give the bits of
the whole product, since the digit sums are exact and the tiles are the same.
The scratch is limited to the least that every product of the call runs with
and to a little more, so that rows of both sides are split, with remainders;
without any the call runs on the FP64 pipe."""
import numpy as np
import pytest

from paper_2304_05505_gb300 import cells

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def thc(cuda_required):
    import os

    from paper_2304_05505_gb300 import build_lib, thc as mod
    if not os.path.exists(mod.LIB_PATH):
        build_lib.build()
    mod.load()
    yield mod
    mod.thc_debug_limit_scratch(-1)


def _least(thc, products):
    """The least scratch with which every one of the products (M, N, K, batch, real) runs."""
    most = 0
    for p in products:
        lo, hi = 0, 1 << 40
        while lo + 1 < hi:
            mid = (lo + hi) // 2
            if thc.thc_debug_slab_plan(*p, mid) is None:
                lo = mid
            else:
                hi = mid
        most = max(most, hi)
    return most


def _limited(thc, call, products):
    """The results of call() with all of the scratch, with little of it, and without."""
    least = _least(thc, products)
    out = []
    try:
        for b in (-1, least, int(1.4 * least), 2 * least, 5 * least, 0):
            thc.thc_debug_limit_scratch(b)
            out.append([np.array(x) for x in call()])
    finally:
        thc.thc_debug_limit_scratch(-1)
    return out


@pytest.mark.parametrize("mesh,nbas,nocc,nisdf", [
    ((2, 2, 1), 90, 70, 301),     # A or B embedded, rows of both sides split
    ((3, 1, 1), 33, 20, 160),     # whole entries and single ones
    ((1, 1, 1), 260, 129, 420),
])
def test_build_in_slabs(thc, mesh, nbas, nocc, nisdf):
    r = cells.random_problem(mesh, nbas=nbas, nocc=nocc, nisdf=nisdf, seed=nisdf)
    nk = int(np.prod(mesh))
    eb = thc.ExchangeBuild(dict(n1=mesh[0], n2=mesh[1], n3=mesh[2], nbas=nbas, nocc=nocc, nisdf=nisdf), "fp64")
    eb.set_collocation(r["X"])
    eb.set_kernel(r["V"])

    def call():
        KC, ex = eb.build(r["C"])
        K, _ = eb.build_K(r["C"])
        eb.sync()
        return KC.cpu().numpy(), ex.cpu().numpy(), K.cpu().numpy()

    try:
        out = _limited(thc, call, [(nisdf, nocc, nbas, nk, 0), (nisdf, nisdf, nocc, nk, 0), (nisdf, nocc, nisdf, nk, 0),
                                   (nbas, nocc, nisdf, nk, 0), (nbas, nisdf, nisdf, nk, 0), (nbas, nbas, nisdf, nk, 0)])
    finally:
        eb.close()
    for got in out[1:-1]:
        for a, b in zip(out[0], got):
            assert np.array_equal(a, b)
    for a, b in zip(out[0], out[-1]):
        assert np.abs(a - b).max() <= 1e-13 * np.abs(a).max()


def test_fit_and_gradient_in_slabs(thc):
    rng = np.random.default_rng(5)
    grid, mesh, nk, nocc, nvir, npts = (9, 11, 10), (1, 2, 1), 2, 20, 13, 130
    ng = int(np.prod(grid))
    nf = nk * nocc
    U = torch.from_numpy(rng.normal(size=(nf, ng)) + 1j * rng.normal(size=(nf, ng))).cuda()
    Uv = torch.from_numpy(rng.normal(size=(nk * nvir, ng)) + 1j * rng.normal(size=(nk * nvir, ng))).cuda()
    lat = np.diag([5.0, 6.0, 7.0])
    pts = np.sort(rng.permutation(ng)[:npts])
    V0 = thc.thc_fit_kernel(U, grid, lat, mesh, pts)
    nG = 9 * 11 * 9

    def call():
        V, xi = thc.thc_fit_kernel(U, grid, lat, mesh, pts, want_xi=True)
        g, ge, ex, _ = thc.thc_vo_gradient(U, Uv, nk, grid, lat, mesh, pts, V0, "fp64")
        return V.cpu().numpy(), xi.cpu().numpy(), g.cpu().numpy(), ge.cpu().numpy(), np.float64(ex)

    out = _limited(thc, call, [(npts, ng, nf, 1, 0), (npts, npts, nG, 1, 0), (npts, npts, nocc, nk, 0),
                               (npts, nocc, npts, nk, 0), (nvir, nocc, npts, nk, 0), (npts, nG, npts, 1, 0),
                               (npts, npts, ng, 1, 1), (npts, nf, ng, 1, 0), (nf, ng, npts, 1, 0),
                               (nvir, nocc, ng, nk, 0), (npts, ng, npts, 1, 1)])
    for got in out[1:-1]:
        for a, b in zip(out[0], got):
            assert np.array_equal(a, b)
    for a, b in zip(out[0], out[-1]):
        assert np.abs(a - b).max() <= 1e-10 * np.abs(a).max()


def test_selection_in_slabs(thc):
    """The Gram matrix of the set, its earlier rows (added with a sign) and the block's rows for every candidate."""
    rng = np.random.default_rng(2)
    nf, nr, npts = 300, 5000, 130
    U = (rng.normal(size=(nf, nr)) + 1j * rng.normal(size=(nf, nr))) * np.exp(0.5 * rng.normal(size=(1, nr)))
    Ud = torch.from_numpy(U).cuda()

    def call():
        pts, resid = thc.thc_select_points(Ud, npts)
        return pts, resid.cpu().numpy()

    out = _limited(thc, call, [(800, 800, nf, 1, 0), (800, 800, npts, 1, 1), (40, nr, npts, 1, 1), (80, 80, nf, 1, 0)])
    for got in out[1:-1]:
        assert np.array_equal(out[0][0], got[0]) and np.array_equal(out[0][1], got[1])
    assert np.array_equal(out[0][0], out[-1][0])     # single pivots
    assert np.abs(out[0][1] - out[-1][1]).max() <= 1e-12 * float(((np.abs(U) ** 2).sum(0) ** 2).max())
