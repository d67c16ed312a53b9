"""Point selection where blocks of pivots do not pay (csrc/pivchol.cu): more than
800 candidates whose densities lie within a bin of the histogram (1/256 octave),
at the start of the selection or with others far below them, so that single
pivots and blocks alternate.  The points are the oracle's, the residuals within
1e-10 of each candidate's own diagonal entry."""
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


@pytest.mark.parametrize("nf,flat,rest,npts", [
    (420, 2400, 0, 70),        # flat throughout
    (420, 801, 1600, 40),      # one more than a set holds
    (12, 900, 83000, 130),     # rank 144: flat at first, then blocks over the rest
    (30, 1000, 34000, 200),
])
def test_flat_top(thc, nf, flat, rest, npts):
    rng = np.random.default_rng(nf + flat)
    n = flat + rest
    U = np.exp(2j * np.pi * rng.uniform(size=(nf, n))) * (1.0 + 1e-5 * rng.uniform(size=n))
    U[:, flat:] *= np.exp(rng.normal(size=rest) * 0.5 - 2.5)
    U = np.ascontiguousarray(U[:, rng.permutation(n)])
    ref = S.pivoted_cholesky(U, npts)
    pts, resid = thc.thc_select_points(torch.from_numpy(U).cuda(), npts)
    assert np.array_equal(pts, ref["points"])
    own = (np.abs(U) ** 2).sum(0) ** 2
    assert (np.abs(resid.cpu().numpy() - ref["resid"]) <= 1e-10 * own).all()
