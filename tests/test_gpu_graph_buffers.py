"""The captured tensor-core build (build_tc_graph, csrc/thc_abi.cu) with buffers
that it cannot serve from one capture, and after builds of another form.  The
results are the bits of a profiled build, whose kernels are launched one by one.
The legacy default stream cannot be captured, so these run on one of their own."""
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
    return mod


@pytest.fixture(autouse=True)
def side_stream(cuda_required):
    with torch.cuda.stream(torch.cuda.Stream()):
        yield
    torch.cuda.synchronize()


def _problem(thc, mesh, nbas, nocc, nisdf, seed):
    r = cells.random_problem(mesh, nbas=nbas, nocc=nocc, nisdf=nisdf, seed=seed)
    eb = thc.ExchangeBuild(dict(n1=mesh[0], n2=mesh[1], n3=mesh[2], nbas=nbas, nocc=nocc, nisdf=nisdf), "mixed")
    eb.set_collocation(r["X"])
    eb.set_kernel(r["V"])
    return eb, torch.from_numpy(np.array(r["C"])).cuda()


def _direct(thc, eb, C):
    thc.thc_profile_begin(eb.ctx, 1)
    KC, _ = eb.build(C)
    thc.thc_profile_end(eb.ctx)
    return KC.cpu()


@pytest.mark.parametrize("mesh,nbas,nocc,nisdf", [
    ((1, 1, 1), 60, 6, 2200),     # K of S4b in chunks: the sum of the chunks stores 32 bytes at a time
    ((2, 1, 1), 33, 5, 40),
    ((1, 1, 1), 6400, 3, 24),     # C is read at its own address
])
def test_alternating_alignments_and_buffers(thc, mesh, nbas, nocc, nisdf):
    eb, C = _problem(thc, mesh, nbas, nocc, nisdf, nisdf)
    try:
        n = int(np.prod(eb.kc_shape))
        other = C * 0.5
        ref = {0: _direct(thc, eb, C), 1: _direct(thc, eb, other)}
        pool = [torch.zeros(n + 2, dtype=torch.complex128, device="cuda") for _ in range(2)]
        for which, buf, off in [(0, 0, 0), (0, 0, 0), (0, 0, 1), (0, 0, 1), (1, 1, 1), (0, 1, 0), (1, 1, 0), (1, 0, 1),
                                (0, 0, 0)]:
            KC = pool[buf][off:off + n].view(eb.kc_shape)
            assert (KC.data_ptr() & 31) == 16 * off
            KC.fill_(7.0)
            eb.build((C, other)[which], KC)
            eb.sync()
            assert torch.equal(KC.cpu(), ref[which])
            assert (pool[buf][n + 1:] == 0).all()
    finally:
        eb.close()


@pytest.mark.parametrize("host", [False, True])
def test_intermediates_of_a_replay_after_another_form(thc, host):
    """Hermitian V: a replayed build writes D on and above the diagonal only;
    thc_build_K writes all of it, with other coefficients here."""
    eb, C = _problem(thc, (2, 2, 2), 30, 5, 64, 3)
    Ch, KCh = C.cpu().pin_memory(), torch.empty(eb.kc_shape, dtype=torch.complex128).pin_memory()
    exh = torch.empty(2, dtype=torch.float64).pin_memory()

    def build():
        if host:
            thc.thc_build_host(eb.ctx, Ch, KCh, exh)
        else:
            eb.build(C)

    try:
        build()
        eb.build_K(C * 2.0)
        build()
        eb.sync()
        Psi, D = (eb.intermediate(i).cpu().numpy() for i in (0, 1))
    finally:
        eb.close()
    ref = np.einsum("kpi,kqi->kpq", Psi, Psi.conj())
    assert np.abs(D - ref).max() <= 1e-5 * np.abs(ref).max()
