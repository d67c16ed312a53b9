"""Scratch that a setup call takes only for speed does not make it fail.

The test hook lets each allocation of the call in turn fail as if the device
were full.  While the call holds scratch for digits it has to give that back and
finish on the FP64 pipe, with the results of the undisturbed call to FP64
accuracy (1e-11 of the largest entry: the sums of the metric change by 1e-15 and
cond(S) is below 1e3 for these unstructured orbitals).  The few allocations
before the scratch is taken end the call with THC_ERR_OOM and leave nothing
behind."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

GRID, MESH, NK, NOCC, NVIR, NPTS = (9, 11, 10), (1, 2, 1), 2, 20, 13, 130


@pytest.fixture(scope="module")
def thc(cuda_required):
    import os

    from paper_2304_05505_gb300 import build_lib, thc as mod
    if not os.path.exists(mod.LIB_PATH):
        build_lib.build()
    mod.load()
    yield mod
    mod.thc_debug_fail_alloc(-1)


def _calls(thc):
    rng = np.random.default_rng(5)
    ng = int(np.prod(GRID))
    U = torch.from_numpy(rng.normal(size=(NK * NOCC, ng)) + 1j * rng.normal(size=(NK * NOCC, ng))).cuda()
    Uv = torch.from_numpy(rng.normal(size=(NK * NVIR, ng)) + 1j * rng.normal(size=(NK * NVIR, ng))).cuda()
    lat, pts = np.diag([5.0, 6.0, 7.0]), np.sort(rng.permutation(ng)[:NPTS])
    V = thc.thc_fit_kernel(U, GRID, lat, MESH, pts)

    def gradient(precision):
        g, ge, _, _ = thc.thc_vo_gradient(U, Uv, NK, GRID, lat, MESH, pts, V, precision)
        return g, ge

    return {
        "fit": lambda: thc.thc_fit_kernel(U, GRID, lat, MESH, pts, want_xi=True),
        "rebuild": lambda: thc.thc_rebuild_kernel(U, GRID, lat, MESH, pts, "fp64")[:1],
        "gradient": lambda: gradient("fp64"),
        "gradient_mixed": lambda: gradient("mixed"),
    }


# (mixed: the operands of its contractions are rounded to FP32, 6e-8)
@pytest.mark.parametrize("name,bound,before", [("fit", 1e-11, 6), ("rebuild", 1e-11, 6), ("gradient", 1e-11, 16),
                                               ("gradient_mixed", 1e-6, 16)])
def test_scratch_is_given_back(thc, name, bound, before):
    call = _calls(thc)[name]
    ref = [x.cpu().numpy() for x in call()]
    failed = []
    for nth in range(40):
        torch.cuda.synchronize()
        free0, _ = torch.cuda.mem_get_info()
        thc.thc_debug_fail_alloc(nth)
        try:
            got = [x.cpu().numpy() for x in call()]
        except thc.ThcError as e:
            assert e.code == 2
            torch.cuda.synchronize()
            assert torch.cuda.mem_get_info()[0] == free0
            failed.append(nth)
            continue
        finally:
            thc.thc_debug_fail_alloc(-1)
        for a, b in zip(ref, got):
            assert np.abs(a - b).max() <= bound * np.abs(a).max(), nth
    assert failed == list(range(before))      # the allocations before the scratch is taken
