"""The forms of the mixed build's convolution that the mesh, the parity of N_P
and the Hermitian symmetry of V choose between, at the sizes where they can go
wrong, against the FP64 oracle.

Bounds: M as a fraction of its largest entry 2e-6 and K C 1e-6 (the mixed
build's bounds on small cells: operands rounded to FP32, 6e-8, a few roundings
deep); the row exponents of M are whole numbers and exact."""
import numpy as np
import pytest

from oracle import thc_oracle as O
from paper_2304_05505_gb300 import cells

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def thc(cuda_required):
    import os

    from paper_2304_05505_gb300 import build_lib, thc as mod
    if not os.path.exists(mod.LIB_PATH):
        build_lib.build()
    mod.load()
    return mod


@pytest.mark.parametrize("mesh,nocc,nisdf", [
    # even N_P, axes of 1, 2, 3, 4, 6 points: tiles of 4 x 8 elements on and above the diagonal
    ((3, 2, 4), 3, 2),        # one tile, most of it outside
    ((6, 4, 2), 3, 10),       # an odd number of row bands, a short last column tile
    ((6, 6, 6), 2, 34),
    ((1, 6, 3), 4, 98),       # just past one square of 12 x 12 blocks of 8 x 8
    ((2, 2, 3), 5, 196),      # two squares and a half
    ((4, 4, 1), 4, 68),
    ((1, 1, 1), 4, 66),
    ((6, 2, 2), 1, 100),      # N_P above 48 n_occ: the keys do not fit, the flat form
    ((5, 2, 4), 3, 12),       # an axis of 5 points: the flat form, rows shorter than its batch
    # odd N_P: M in padded rows
    ((3, 2, 4), 3, 33),
    ((4, 4, 4), 2, 7),
    ((3, 3, 3), 2, 1),
    ((2, 2, 2), 3, 51),
    ((5, 1, 2), 4, 129),
    ((7, 8, 1), 2, 13),
])
@pytest.mark.parametrize("hermitian", [True, False])
def test_convolution_forms(thc, mesh, nocc, nisdf, hermitian):
    r = cells.random_problem(mesh, nbas=9, nocc=nocc, nisdf=nisdf, seed=nisdf + 3)
    V = r["V"]
    if not hermitian:
        rng = np.random.default_rng(nisdf)
        V = V + 0.05 * np.abs(V).max() * (rng.normal(size=V.shape) + 1j * rng.normal(size=V.shape))
    ref = O.build(r["X"], r["C"], V, r["mesh"], keep=True)
    dims = dict(n1=mesh[0], n2=mesh[1], n3=mesh[2], nbas=9, nocc=nocc, nisdf=nisdf)
    eb = thc.ExchangeBuild(dims, "mixed")
    try:
        eb.set_collocation(r["X"])
        eb.set_kernel(V)
        KC, _ = eb.build(r["C"])
        eb.sync()
        KC = KC.cpu().numpy()
        M, D = eb.intermediate(2).cpu().numpy(), eb.intermediate(1).cpu().numpy()
        eM = eb.intermediate(4).cpu().numpy()
        KC2, _ = eb.build(r["C"])
        assert np.array_equal(KC2.cpu().numpy(), KC)
    finally:
        eb.close()
    assert np.abs(KC - ref["KC"]).max() <= 1e-6 * np.abs(ref["KC"]).max()
    assert np.abs(M - ref["M"]).max() <= 2e-6 * np.abs(ref["M"]).max()
    assert np.abs(D - ref["D"]).max() <= 2e-6 * np.abs(ref["D"]).max()
    m = np.maximum(np.abs(M.real), np.abs(M.imag)).max(axis=2)
    assert np.array_equal(eM, np.where(m > 0, np.frexp(m)[1], 0).astype(np.float64))
