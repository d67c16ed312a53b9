"""What an FP64 context holds and reports: its memory, its intermediates (D
serves as scratch once the convolution has read it), its stage times and the
bounded waits of its products."""
import numpy as np
import pytest

from oracle import thc_oracle as O
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
    return mod


def _context(thc, mesh, nbas, nocc, nisdf):
    return thc.ExchangeBuild(dict(n1=mesh[0], n2=mesh[1], n3=mesh[2], nbas=nbas, nocc=nocc, nisdf=nisdf), "fp64")


@pytest.mark.parametrize("mesh,nbas,nocc,nisdf,extra", [((4, 4, 4), 216, 30, 900, 0), ((1, 1, 1), 300, 60, 900, 512)])
def test_memory_is_what_the_library_says(thc, mesh, nbas, nocc, nisdf, extra):
    """After the inputs are set and a build has run, the device holds no more
    than thc_memory_bytes, the 512 MB that contexts with a D below that may
    take, and 2 MB of rounding for each of at most 16 allocations."""
    nk = int(np.prod(mesh))
    X, C, V = (torch.randn(nk, *s, dtype=torch.complex128, device="cuda")
               for s in ((nbas, nisdf), (nbas, nocc), (nisdf, nisdf)))
    KC, ex = torch.empty_like(C), torch.empty(2, dtype=torch.float64, device="cuda")
    _context(thc, (2, 1, 1), 40, 20, 200).close()      # the library's own modules are loaded
    w = _context(thc, mesh, nbas, nocc, nisdf)
    w.set_collocation(X)
    w.set_kernel(V)
    w.build(C, KC, ex)
    w.sync()
    w.close()
    torch.cuda.synchronize()
    free0, _ = torch.cuda.mem_get_info()
    eb = _context(thc, mesh, nbas, nocc, nisdf)
    try:
        eb.set_collocation(X)
        eb.set_kernel(V)
        eb.build(C, KC, ex)
        eb.sync()
        free1, _ = torch.cuda.mem_get_info()
    finally:
        eb.close()
    own = thc.thc_memory_bytes(dict(n1=mesh[0], n2=mesh[1], n3=mesh[2], nbas=nbas, nocc=nocc, nisdf=nisdf), thc.THC_FP64)
    assert free0 - free1 <= own + (extra << 20) + (32 << 20)


@pytest.mark.parametrize("mesh,nbas,nocc,nisdf", [((3, 2, 2), 40, 33, 129), ((1, 1, 2), 130, 41, 333)])
def test_intermediates_after_builds(thc, mesh, nbas, nocc, nisdf):
    """D, M and the rest of both builds against the oracle (1e-13 of the
    largest entry: each product rounds once, as in test_gpu_digits.py), also
    asked for twice, and stage times in their slots."""
    r = cells.random_problem(mesh, nbas=nbas, nocc=nocc, nisdf=nisdf, seed=2)
    ref = O.build(r["X"], r["C"], r["V"], r["mesh"], route="direct", keep=True)
    eb = _context(thc, mesh, nbas, nocc, nisdf)
    try:
        eb.set_collocation(r["X"])
        eb.set_kernel(r["V"])
        for call in (eb.build, eb.build_K, eb.build):
            _, ex = call(r["C"])
            eb.sync()
            assert abs(float(ex[0]) - ref["Ex"]) <= 1e-13 * abs(ref["Ex"])
            for _ in range(2):
                for i, name in ((1, "D"), (2, "M")):
                    got = eb.intermediate(i).cpu().numpy()
                    assert np.abs(got - ref[name]).max() <= 1e-13 * np.abs(ref[name]).max(), (call.__name__, name)
            assert all(t > 0 for t in thc.thc_stage_times(eb.ctx))
    finally:
        eb.close()


def test_wait_timeout_of_products_is_reported(thc):
    """A limit of a few hundred cycles lets the waits of the digit products
    give up before their data arrive; thc_sync says so, and with the default
    limit the context builds correctly again."""
    mesh, nbas, nocc, nisdf = (2, 2, 2), 60, 33, 260
    r = cells.random_problem(mesh, nbas=nbas, nocc=nocc, nisdf=nisdf, seed=3)
    ref = O.build(r["X"], r["C"], r["V"], mesh, route="direct")
    eb = _context(thc, mesh, nbas, nocc, nisdf)
    try:
        eb.set_collocation(r["X"])
        eb.set_kernel(r["V"])
        thc.thc_debug_set_wait_limit(eb.ctx, 200)
        eb.build(r["C"])
        with pytest.raises(thc.ThcError) as e:
            eb.sync()
        assert e.value.code == 5                      # THC_ERR_TIMEOUT
        thc.thc_debug_set_wait_limit(eb.ctx, 0)
        KC, ex = eb.build(r["C"])
        eb.sync()
        assert np.abs(KC.cpu().numpy() - ref["KC"]).max() <= 1e-13 * np.abs(ref["KC"]).max()
    finally:
        thc.thc_debug_set_wait_limit(eb.ctx, 0)
        eb.close()
