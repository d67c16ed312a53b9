"""bench.py's rule for the tiled Hermitian convolution (csrc/thc_abi.cu, herm_tile_form)."""
import pytest

import bench


def _dims(mesh, nocc, nisdf):
    return dict(n1=mesh[0], n2=mesh[1], n3=mesh[2], nbas=4 * nocc, nocc=nocc, nisdf=nisdf)


@pytest.mark.parametrize("mesh,nocc,nisdf,tiled", [
    ((6, 6, 6), 120, 2400, True),      # C3
    ((3, 2, 4), 23, 702, True),
    ((3, 2, 4), 23, 701, False),       # odd N_P: D's rows are not 16-byte strided
    ((5, 3, 2), 23, 702, False),       # an axis of 5 points
    ((6, 6, 6), 10, 2400, False),      # the keys do not fit the planes
    ((6, 6, 6), 60, 2400, True),
])
def test_hermitian_tiles_rule(mesh, nocc, nisdf, tiled):
    assert bench.hermitian_tiles(_dims(mesh, nocc, nisdf)) is tiled


def test_work_of_the_tiled_form_is_the_hermitian_one():
    names = bench.kernel_names(False, True)
    assert "kconv_tile_herm_kernel" in names["S3_kconv"]
    assert "mirrored" not in names["S2_density"]
