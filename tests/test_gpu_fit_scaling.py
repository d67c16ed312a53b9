"""The fit does not depend on the scale of the density at a point.

With the orbitals' values at grid point r multiplied by s_r, R[P][r] and S[P][Q]
take the factors (s_P s_r)^2 and (s_P s_Q)^2, so xi = S^-1 R takes (s_r / s_P)^2.
For powers of two every product, square, pivot and substitution of the scaled
fit is the unscaled one times a power of two, so xi has to scale to the bit,
whatever the span: 2^64 (2e19) in the density here."""
import numpy as np
import pytest

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
    (16, (7, 9, 5), 31),
    (33, (16, 16, 16), 41),
    (70, (12, 11, 13), 129),
    (90, (15, 16, 17), 300),
])
def test_fit_scales_with_the_density(thc, nfunc, grid, npts):
    rng = np.random.default_rng(nfunc)
    ng = int(np.prod(grid))
    U = rng.normal(size=(nfunc, ng)) + 1j * rng.normal(size=(nfunc, ng))
    s = 2.0 ** rng.integers(-16, 17, size=ng)
    pts = np.sort(rng.permutation(ng)[:npts])
    lat = np.diag([5.0, 6.0, 7.0])

    def fit(u):
        return thc.thc_fit_kernel(torch.from_numpy(u).cuda(), grid, lat, (1, 1, 1), pts, want_xi=True)[1].cpu().numpy()

    xi = fit(U)
    assert np.array_equal(fit(U * s), xi * (s[None, :] / s[pts][:, None]) ** 2)
