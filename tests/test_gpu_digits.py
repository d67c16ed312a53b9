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
