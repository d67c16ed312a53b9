"""The work that a user of this library has it do, as cases that can be timed.

An SCF iteration of THC-oo-K refits the kernel to its orbitals
(``thc_rebuild_kernel``) and runs the exchange build (``ExchangeBuild.build``,
or from host buffers ``thc_build_host``); the interpolation points are selected
once per geometry (``thc_select_points``), and a gradient-based solver asks for
the orbital gradient (``thc_vo_gradient``).  ``build_K`` is the THC-AO-K form
of the build.  Sizes are those of the synthetic cells of ``cells.py`` (C0 to
C3: the toy cell and the benzene-shaped ones) and generic ones around them.

``kind`` says which call a case makes:

* ``build``, ``host``, ``ao_k``: one exchange build of N_k = n1 n2 n3 points,
  ``nbas`` basis functions, ``nocc`` orbitals and ``nisdf`` points in the form
  ``prec``; ``fresh`` lets the call allocate its outputs, as the README does;
* ``rebuild``, ``select``, ``vo``: the set-up and gradient calls on orbitals
  given on the ``grid`` (g1 x g2 x g3 points).

The inputs are a benzene-shaped orthorhombic cell (scaled with the grid) of
Bloch-summed Cartesian Gaussians at random centres, coefficients that are
smooth in k and obey C^-k = conj(C^k), and kernels that are Hermitian and
positive semidefinite for every q, as an ISDF fit gives them.  They are made on
the GPU from the seed.
"""
import math

import numpy as np
import torch

from paper_2304_05505_gb300 import thc

DEV = "cuda"
CELL = (13.9, 17.8, 12.9)                  # bohr, on 40 x 40 x 40 grid points
C128 = torch.complex128


def _build(name, mesh, nbas, nocc, nisdf, prec="mixed", kind="build", fresh=False):
    n1, n2, n3 = mesh
    return dict(name=name, kind=kind, prec=prec, n1=n1, n2=n2, n3=n3, nbas=nbas, nocc=nocc, nisdf=nisdf, fresh=fresh)


def _grid(name, kind, mesh, grid, nocc, nisdf, nvir=0, prec="mixed"):
    n1, n2, n3 = mesh
    g1, g2, g3 = grid
    return dict(name=name, kind=kind, prec=prec, n1=n1, n2=n2, n3=n3, g1=g1, g2=g2, g3=g3, nocc=nocc, nvir=nvir,
                nisdf=nisdf)


def listed():
    return [
        # the smallest cell (C0): launches and latency are the whole call
        _build("build_toy", (2, 2, 2), 16, 4, 48),
        # the benzene-shaped cell on a 3 x 3 x 3 mesh (C1), the README's call: outputs allocated by the build
        _build("build_c1", (3, 3, 3), 432, 60, 600, fresh=True),
        # the headline workload (C2): 4 x 4 x 4 k
        _build("build_c2", (4, 4, 4), 432, 60, 1200),
        # the largest: a 96-centre supercell on a 6 x 6 x 6 mesh (C3)
        _build("build_c3", (6, 6, 6), 864, 120, 2400),
        # C2 for a code that keeps C and K C on the host (the end-to-end call)
        _build("host_c2", (4, 4, 4), 432, 60, 1200, kind="host"),
        # an anisotropic mesh and ragged sizes: no size is a multiple of anything
        _build("build_ragged", (3, 2, 4), 217, 23, 701, fresh=True),
        # C2 with M carried to 35 bits, for fitted kernels
        _build("build_ext_c2", (4, 4, 4), 432, 60, 1200, prec="mixed_ext"),
        # C2 all in FP64: the reference precision, the last iterations of a tight SCF
        _build("build_fp64_c2", (4, 4, 4), 432, 60, 1200, prec="fp64"),
        # the full AO exchange matrix (THC-AO-K) of C1
        _build("ao_k_c1", (3, 3, 3), 432, 60, 600, kind="ao_k"),
        # every SCF iteration: the kernel refitted to the orbitals of C1
        _grid("rebuild_c1", "rebuild", (3, 3, 3), (40, 40, 40), 60, 600),
        # once per geometry: 600 points by pivoted Cholesky over the whole 40^3 grid
        _grid("select_c1", "select", (3, 3, 3), (40, 40, 40), 60, 600),
        # the orbital gradient with the kernel's response, on a coarser grid
        _grid("vo_grad", "vo", (3, 3, 3), (32, 32, 32), 40, 400, nvir=120),
    ]


def draw(rng):
    def log(a, b):
        return int(round(math.exp(rng.uniform(math.log(a), math.log(b)))))

    kind = rng.choice(["build"] * 8 + ["host", "ao_k", "rebuild", "rebuild", "select", "vo", "vo"])
    if kind in ("build", "host", "ao_k"):
        while True:
            n = rng.choice([(2, 2, 2), (3, 3, 3), (4, 4, 4), (6, 6, 6)] * 2 +
                           [(1, 1, 1), (2, 2, 1), (3, 2, 4), (4, 4, 2), (1, 1, 8), (5, 3, 2), (5, 5, 5)])
            nk = n[0] * n[1] * n[2]
            nocc = log(4, 120)
            nbas = min(864, max(16, int(nocc * rng.uniform(3, 8))))
            nisdf = min(2400, max(48, int(nocc * rng.uniform(8, 22))))
            prec = "mixed" if kind == "host" else rng.choice(
                ["mixed", "mixed", "fp64"] if kind == "ao_k" else ["mixed"] * 5 + ["mixed_ext", "fp64", "fp64"])
            cost = nk * nisdf * (2.0 * nbas * nocc + 2 * nisdf * nocc if kind != "ao_k" else nisdf * nbas + nbas * nbas)
            most = {"mixed": 1.5e11, "mixed_ext": 3e10, "fp64": 1.5e10}[prec] if kind == "build" else 3e10
            if prec == "fp64":
                most = 1.5e10
            if cost <= most:
                break
        c = _build("", n, nbas, nocc, nisdf, prec, kind, fresh=kind == "build" and rng.random() < 0.4)
    else:
        while True:
            n = tuple(rng.choice([1, 2, 2, 3, 3, 4]) for _ in range(3))
            nk = n[0] * n[1] * n[2]
            g = tuple(rng.randint(12, 40) for _ in range(3))
            nocc = log(6, 60)
            nvir = nocc * rng.randint(1, 3) if kind == "vo" else 0
            nisdf = max(24, min(600, int(nocc * rng.uniform(5, 9))))
            ng = g[0] * g[1] * g[2]
            prec = rng.choice(["mixed", "mixed", "fp64"]) if kind != "select" else "fp64"
            reps = np.prod([m if m % 2 else m + 1 for m in n])     # (q, representative) pairs
            fp64 = 1.0 * ng * nk * nocc * nisdf + (ng * nisdf ** 2.0 * reps if prec == "fp64" and kind != "select" else 0)
            if nk >= 2 and ng >= 12 * nisdf and fp64 <= 5e10 and (kind != "vo" or nk * (nocc + nvir) * ng <= 1.5e8):
                break
        c = _grid("", kind, n, g, nocc, nisdf, nvir, prec)
    del c["name"]
    return c


# ----------------------------------------------------------------------------
# inputs
# ----------------------------------------------------------------------------

def _mesh(c):
    return c["n1"], c["n2"], c["n3"]


def _kfrac(n):
    a = [torch.arange(m, dtype=torch.float64, device=DEV) / m for m in n]
    return torch.stack(torch.meshgrid(*a, indexing="ij"), -1).reshape(-1, 3)


class _Rand:
    """Random numbers on the device, from a seed."""

    def __init__(self, seed):
        self.g = torch.Generator(device=DEV).manual_seed(1000003 * int(seed) + 17)

    def normal(self, *s):
        return torch.randn(s, generator=self.g, dtype=torch.float64, device=DEV)

    def uniform(self, *s):
        return torch.rand(s, generator=self.g, dtype=torch.float64, device=DEV)

    def integers(self, n, *s):
        return torch.randint(n, s, generator=self.g, device=DEV)


def _basis(r, cell, nbas):
    """nbas Cartesian Gaussians x^l y^m z^n exp(-a |r - A|^2), normalised to about one: centres near
    nbas / 9 atoms, exponents 0.25 to 3.5 bohr^-2, s, p and d powers."""
    atoms = r.uniform(max(4, nbas // 9), 3) * cell
    centre = atoms[r.integers(atoms.shape[0], nbas)] + 0.05 * r.normal(nbas, 3)
    alpha = torch.exp(r.uniform(nbas) * math.log(3.5 / 0.25)) * 0.25
    powers = torch.tensor([[0, 0, 0]] * 3 + [[1, 0, 0], [0, 1, 0], [0, 0, 1]] * 2 + [[1, 1, 0], [0, 1, 1], [1, 0, 1]],
                          device=DEV)[r.integers(12, nbas)]
    norm = (2 * alpha / math.pi) ** 0.75 * (4 * alpha) ** (powers.sum(1) / 2)
    return centre, alpha, powers, norm


def _axis_bloch(x, k, length, centre, alpha, power, periodic):
    """sum_R exp(i k R) (x - A - R)^l exp(-a (x - A - R)^2) for k in turns per cell ([k][function][point]); times
    exp(-i k x) when `periodic` (the cell-periodic part)."""
    out = torch.zeros((k.shape[0], centre.shape[0], x.shape[-1]), dtype=C128, device=DEV)
    for n in range(-2, 3):
        d = x - centre[:, None] - n * length
        v = torch.where(power[:, None] == 1, d, torch.ones_like(d)) * torch.exp(-alpha[:, None] * d * d)
        out += torch.exp(2j * math.pi * k * n)[:, None, None] * v
    if periodic:
        out *= torch.exp(-2j * math.pi * k[:, None] * (x / length).reshape(1, -1))[:, None, :]
    return out


def _coefficients(r, kf, nbas, norb):
    """C^k = (c0 + sum_a c_a exp(2 pi i k_a)) / sqrt(nbas), c real: smooth in k, C^-k = conj(C^k)."""
    C = r.normal(nbas, norb).to(C128).expand(kf.shape[0], nbas, norb).clone()
    for a in range(3):
        C += 0.4 * torch.exp(2j * math.pi * kf[:, a])[:, None, None] * r.normal(nbas, norb)
    return C / math.sqrt(1.5 * nbas)


def _build_inputs(c, seed):
    """X [N_k][nbas][nisdf], C [N_k][nbas][nocc], V [N_k][nisdf][nisdf] on the device."""
    r, n = _Rand(seed), _mesh(c)
    kf = _kfrac(n)
    nk, P = kf.shape[0], c["nisdf"]
    cell = torch.tensor(CELL, dtype=torch.float64, device=DEV)
    centre, alpha, powers, norm = _basis(r, cell, c["nbas"])
    # points near the centres, where the density is
    pts = (centre[r.integers(c["nbas"], P)] + 1.2 * r.normal(P, 3)) % cell
    X = None
    for a in range(3):
        ka = torch.arange(n[a], dtype=torch.float64, device=DEV) / n[a]
        f = _axis_bloch(pts[:, a], ka, CELL[a], centre[:, a], alpha, powers[:, a], False)
        sel = torch.round(kf[:, a] * n[a]).long()
        X = f[sel] * norm[:, None] if X is None else X.mul_(f[sel])
    C = _coefficients(r, kf, c["nbas"], c["nocc"])
    # V^q = 1/(N_k Omega) sum_K w_P w_Q v(K) exp(-K^2 / 2) exp(-i K.(r_P - r_Q)), K = q + G over a small symmetric
    # set of G, plus a diagonal
    V = torch.empty((nk, P, P), dtype=C128, device=DEV)
    g = torch.arange(-2.0, 3.0, dtype=torch.float64, device=DEV)
    G = torch.stack(torch.meshgrid(g, g, g, indexing="ij"), -1).reshape(-1, 3)
    w = (cell.prod() / P) * (0.5 + r.uniform(P))
    for q in range(nk):
        K = (G + kf[q] - torch.round(kf[q])) * (2 * math.pi / cell)
        k2 = (K * K).sum(1)
        s = torch.where(k2 > 1e-12, 4 * math.pi / k2.clamp(min=1e-12) * torch.exp(-k2 / 2), torch.zeros_like(k2))
        A = torch.exp(-1j * (pts @ K.T)) * torch.sqrt(s / (nk * cell.prod())) * w[:, None]
        W = A @ A.conj().T
        V[q] = 0.5 * (W + W.conj().T)
        V[q].diagonal().add_((w / (nk * cell.prod())).to(C128))
    return X, C, V


def _grid_inputs(c, seed, want_v=False):
    """Orbitals' periodic parts on the grid (U, Uv), points, cell; and the fitted kernel for the gradient."""
    r, n, g = _Rand(seed), _mesh(c), (c["g1"], c["g2"], c["g3"])
    kf = _kfrac(n)
    nk, ng = kf.shape[0], g[0] * g[1] * g[2]
    size = [CELL[a] * g[a] / 40.0 for a in range(3)]
    cell = torch.tensor(size, dtype=torch.float64, device=DEV)
    norb = c["nocc"] + c["nvir"]
    nfun = max(24, 2 * c["nocc"], norb)
    centre, alpha, powers, norm = _basis(r, cell, nfun)
    C = _coefficients(r, kf, nfun, norb)
    f = []
    for a in range(3):
        ka = torch.arange(n[a], dtype=torch.float64, device=DEV) / n[a]
        x = torch.arange(g[a], dtype=torch.float64, device=DEV) * (size[a] / g[a])
        f.append(_axis_bloch(x, ka, size[a], centre[:, a], alpha, powers[:, a], True))
    U = torch.empty((nk, c["nocc"], ng), dtype=C128, device=DEV)
    Uv = torch.empty((nk, c["nvir"], ng), dtype=C128, device=DEV)
    for k in range(nk):
        i = [int(round(float(kf[k, a]) * n[a])) for a in range(3)]
        phi = f[0][i[0]][:, :, None, None] * f[1][i[1]][:, None, :, None] * f[2][i[2]][:, None, None, :]
        u = C[k].T @ (phi.reshape(nfun, ng) * norm[:, None])
        U[k], Uv[k] = u[:c["nocc"]], u[c["nocc"]:]
    U, Uv = U.reshape(-1, ng), Uv.reshape(-1, ng)
    lattice = np.diag(size)
    points = _choose_points(r, U, c["nisdf"]) if c["kind"] != "select" else None
    V = _fitted_kernel(c, U, points, lattice, torch.complex64) if want_v else None
    return U, Uv, points, lattice, g, n, V


def _choose_points(r, U, npts):
    """npts grid points: pivoted Cholesky of the pair Gram matrix over 4 npts candidates drawn by density."""
    rho = (U.real ** 2 + U.imag ** 2).sum(0)
    cand = torch.multinomial(rho + 0.02 * rho.mean(), min(4 * npts, U.shape[1]), generator=r.g)
    cand = torch.sort(cand).values
    Uc = U[:, cand]
    A = (Uc.conj().T @ Uc).abs() ** 2
    d, L, got = A.diagonal().clone(), torch.zeros((npts, cand.shape[0]), dtype=torch.float64, device=DEV), []
    for j in range(npts):
        p = torch.argmax(d).reshape(1)
        got.append(p)
        col = A.index_select(0, p)[0] - L.index_select(1, p)[:, 0] @ L
        L[j] = col / torch.sqrt(d.index_select(0, p))
        d = torch.clamp(d - L[j] ** 2, min=0).index_fill(0, p, 0.0)
    return cand[torch.cat(got)].cpu().numpy()


# ----------------------------------------------------------------------------
# the calls
# ----------------------------------------------------------------------------

def prepare(case, seed):
    c = dict(case)
    if c["kind"] in ("build", "host", "ao_k"):
        X, C, V = _build_inputs(c, seed)
        dims = {k: c[k] for k in ("n1", "n2", "n3", "nbas", "nocc", "nisdf")}
        eb = thc.ExchangeBuild(dims, c["prec"])
        eb.set_collocation(X)
        eb.set_kernel(V)
        nk = X.shape[0]
        del X, V
        torch.cuda.empty_cache()               # the context's memory is its own; the inputs are not kept
        s = dict(c, eb=eb, C=C, out=None, ex=None)
        if c["kind"] == "host":
            s["C"] = C.cpu().pin_memory()
            s["out"] = torch.empty_like(s["C"]).pin_memory()
            s["ex"] = torch.empty(2, dtype=torch.float64).pin_memory()
        elif not c["fresh"]:
            cols = c["nbas"] if c["kind"] == "ao_k" else c["nocc"]
            s["out"] = torch.empty((nk, c["nbas"], cols), dtype=C128, device=DEV)
            s["ex"] = torch.empty(2, dtype=torch.float64, device=DEV)
        return s
    U, Uv, points, lattice, g, n, V = _grid_inputs(c, seed, want_v=c["kind"] == "vo")
    return dict(c, U=U, Uv=Uv, points=points, lattice=lattice, grid=g, mesh=n, V=V)


def run(s):
    if s["kind"] == "build":
        return s["eb"].build(s["C"], s["out"], s["ex"])
    if s["kind"] == "ao_k":
        return s["eb"].build_K(s["C"], s["out"], s["ex"])
    if s["kind"] == "host":
        thc.thc_build_host(s["eb"].ctx, s["C"], s["out"], s["ex"])
        return s["out"], s["ex"]
    if s["kind"] == "rebuild":
        return thc.thc_rebuild_kernel(s["U"], s["grid"], s["lattice"], s["mesh"], s["points"], s["prec"])[0]
    if s["kind"] == "select":
        return thc.thc_select_points(s["U"], s["nisdf"])
    nk = s["n1"] * s["n2"] * s["n3"]
    return thc.thc_vo_gradient(s["U"], s["Uv"], nk, s["grid"], s["lattice"], s["mesh"], s["points"], s["V"],
                               s["prec"])[:3]


def work(case):
    """Bytes: each input read once, each output written once, X and V in the context's precision (the upper half of
    the Hermitian V).  Flops: 8 per complex multiply-add of the contractions, and the transforms."""
    c = case
    nk, P, n = c["n1"] * c["n2"] * c["n3"], c["nisdf"], c["nocc"]
    if c["kind"] in ("build", "host", "ao_k"):
        N = c["nbas"]
        el = 16 if c["prec"] == "fp64" else 8
        out = N * N if c["kind"] == "ao_k" else N * n
        back = P * P * N + P * N * N if c["kind"] == "ao_k" else P * P * n + P * N * n
        return {"bytes": float(nk * (el * (N * P + P * (P + 1) // 2) + 16 * (N * n + out))),
                "flops": float(8 * nk * (P * N * n + P * (P + 1) // 2 * n + back)
                               + 5 * nk * P * (P + 1) * max(1.0, math.log2(nk)))}
    ng = c["g1"] * c["g2"] * c["g3"]
    nf = nk * n
    if c["kind"] == "select":
        # the points' Gram columns, and the triangular elimination
        return {"bytes": 16.0 * nf * ng + 8 * ng, "flops": 8.0 * nf * ng * P + ng * P ** 2.0}
    nG = np.prod([2 * ((c[a] - 1) // 2) + 1 for a in ("g1", "g2", "g3")])
    fit = 8.0 * nf * ng * P + P ** 3 / 3.0 + 2.0 * ng * P ** 2 + 5 * P * ng * math.log2(ng)
    if c["kind"] == "rebuild":      # fit, and the Hermitian contraction of every q
        return {"bytes": 16.0 * nf * ng + 16.0 * nk * P * P, "flops": float(fit + 4.0 * nk * P * P * nG)}
    nv = nk * c["nvir"]
    grad = 8.0 * nk * P * P * nG + 2.0 * ng * P ** 2 + 16.0 * nf * ng * P + 8.0 * nv * n * ng
    return {"bytes": 16.0 * (nf + nv) * ng + 16.0 * nk * P * P + 32.0 * nv * n, "flops": float(fit + grad)}


# ----------------------------------------------------------------------------
# the same in plain torch, in 64 bits
# ----------------------------------------------------------------------------

def exact(case, seed):
    c = dict(case)
    if c["kind"] in ("build", "host", "ao_k"):
        return _exact_build(c, seed)
    U, Uv, points, lattice, g, n, V = _grid_inputs(c, seed, want_v=c["kind"] == "vo")
    if c["kind"] == "select":
        return [None, _exact_residual(U, c["nisdf"])]
    if c["kind"] == "rebuild":
        return _fitted_kernel(c, U, points, lattice, C128)
    return _exact_gradient(c, U, Uv, points, lattice, V)


def _exact_build(c, seed):
    X, C, V = _build_inputs(c, seed)
    n, nk, P = _mesh(c), X.shape[0], c["nisdf"]
    Psi = X.transpose(1, 2) @ C
    D = Psi @ Psi.conj().transpose(1, 2)
    M = torch.empty_like(D)
    step = max(1, int(2e8 // (nk * P)))
    for p in range(0, P, step):                # rows at a time: M^k = sum_k' D^k' o V^(k' - k) by FFT over the mesh
        d = torch.fft.fftn(D[:, p:p + step].reshape(n + (-1, P)), dim=(0, 1, 2))
        v = torch.fft.ifftn(V[:, p:p + step].reshape(n + (-1, P)), dim=(0, 1, 2)) * nk
        M[:, p:p + step] = torch.fft.ifftn(d.mul_(v), dim=(0, 1, 2)).reshape(nk, -1, P)
    del V
    if c["kind"] == "ao_k":
        out = X.conj() @ (M @ X.transpose(1, 2))
        e = torch.stack([(D[k].conj() * M[k]).sum() for k in range(nk)]).sum()
    else:
        Y = M @ Psi
        out, e = X.conj() @ Y, (Psi.conj() * Y).sum()
    return [out, torch.view_as_real(-e / nk).clone()]


def _exact_residual(U, npts):
    """Residual diagonal of the pivoted Cholesky of |U^H U|^2 after npts points."""
    d = (U.real ** 2 + U.imag ** 2).sum(0) ** 2
    L = torch.zeros((npts, U.shape[1]), dtype=torch.float64, device=DEV)
    for j in range(npts):
        p = torch.argmax(d).reshape(1)
        col = (U.index_select(1, p)[:, 0].conj() @ U).abs() ** 2 - L.index_select(1, p)[:, 0] @ L
        L[j] = col / torch.sqrt(d.index_select(0, p))
        d = torch.clamp(d - L[j] ** 2, min=0).index_fill(0, p, 0.0)
    return d


def _gvectors(g):
    a = [torch.arange(-((m - 1) // 2), (m - 1) // 2 + 1, device=DEV) for m in g]
    G = torch.stack(torch.meshgrid(*a, indexing="ij"), -1).reshape(-1, 3)
    flat = ((G[:, 0] % g[0]) * g[1] + G[:, 1] % g[1]) * g[2] + G[:, 2] % g[2]
    return G.to(torch.float64), flat


def _shifts(n):
    """(q index, q in turns, weight) of every minimum-image representative of every q."""
    def axis(i, m):
        f = i / m
        return [0.5, -0.5] if abs(f - 0.5) < 1e-12 else [f - 1] if f > 0.5 else [f]

    for q in range(n[0] * n[1] * n[2]):
        i = (q // (n[1] * n[2]), (q // n[2]) % n[1], q % n[2])
        reps = [(a, b, d) for a in axis(i[0], n[0]) for b in axis(i[1], n[1]) for d in axis(i[2], n[2])]
        for t in reps:
            yield q, t, 1.0 / len(reps)


class _Fit:
    """xi = S^-1 R, its transform, and the pieces the kernel and its adjoint share."""

    def __init__(self, c, U, points, lattice):
        self.g, self.n = (c["g1"], c["g2"], c["g3"]), _mesh(c)
        self.p = torch.as_tensor(points, device=DEV)
        self.len = torch.tensor(np.diag(lattice), dtype=torch.float64, device=DEV)
        self.vol = float(self.len.prod())
        ng = U.shape[1]
        self.B = U[:, self.p].conj().T @ U
        R = self.B.real ** 2 + self.B.imag ** 2
        self.S = R[:, self.p]
        self.S = 0.5 * (self.S + self.S.T)
        self.L = torch.linalg.cholesky(self.S)
        self.xi = torch.cholesky_solve(R, self.L)
        self.G, self.flat = _gvectors(self.g)
        self.xh = torch.fft.fftn(self.xi.reshape((-1,) + self.g).to(C128), dim=(1, 2, 3)).reshape(-1, ng)[:, self.flat]
        self.xh *= self.vol / ng
        r = torch.stack([self.p // (self.g[1] * self.g[2]), (self.p // self.g[2]) % self.g[1], self.p % self.g[2]], 1)
        self.rf = r.to(torch.float64) / torch.tensor(self.g, dtype=torch.float64, device=DEV)

    def coulomb(self, t):
        K = (self.G + torch.tensor(t, dtype=torch.float64, device=DEV)) * (2 * math.pi / self.len)
        k2 = (K * K).sum(1)
        return torch.where(k2 > 1e-12, 4 * math.pi / k2.clamp(min=1e-12), torch.zeros_like(k2))

    def phase(self, t):
        return torch.exp(-2j * math.pi * (self.rf @ torch.tensor(t, dtype=torch.float64, device=DEV)))


def _fitted_kernel(c, U, points, lattice, dtype):
    f = _Fit(c, U, points, lattice)
    nk, P = f.n[0] * f.n[1] * f.n[2], len(points)
    V = torch.zeros((nk, P, P), dtype=C128, device=DEV)
    for q, t, w in _shifts(f.n):
        A = (f.xh * torch.sqrt(f.coulomb(t) * w / (nk * f.vol)) * f.phase(t)[:, None]).to(dtype)
        W = A @ A.conj().T
        V[q] += (0.5 * (W + W.conj().T)).to(C128)
    return V


def _exact_gradient(c, U, Uv, points, lattice, V):
    """The derivative of E_x for C -> C + Cv theta, by the adjoint of the fit (V given)."""
    f, n = _Fit(c, U, points, lattice), _mesh(c)
    nk, P, no, nv, ng = V.shape[0], len(points), c["nocc"], c["nvir"], U.shape[1]
    kf = _kfrac(n)
    bloch = torch.exp(2j * math.pi * (kf @ f.rf.T))                                   # [k][P]
    Psi = U[:, f.p].reshape(nk, no, P).transpose(1, 2) * bloch[:, :, None]
    Psiv = Uv[:, f.p].reshape(nk, nv, P).transpose(1, 2) * bloch[:, :, None]
    D = Psi @ Psi.conj().transpose(1, 2)
    fd = torch.fft.fftn(D.reshape(n + (P, P)), dim=(0, 1, 2))
    W = torch.fft.ifftn(fd.abs() ** 2, dim=(0, 1, 2)).reshape(nk, P, P)               # sum_k conj(D^k) D^(k+q)
    M = torch.fft.ifftn(fd * torch.fft.ifftn(V.reshape(n + (P, P)), dim=(0, 1, 2)) * nk, dim=(0, 1, 2))
    Y = M.reshape(nk, P, P) @ Psi
    ge = -(4.0 / nk) * (Psiv.conj().transpose(1, 2) @ Y)
    ex = -float((W * V).sum().real) / nk
    gam = torch.zeros_like(f.xh)
    for q, t, w in _shifts(n):
        ph = f.phase(t)
        A = (-2.0 / nk * (f.vol / ng) * w / (nk * f.vol)) * ph[:, None] * W[q] * ph.conj()
        gam += A @ (f.coulomb(t) * f.xh.conj())
    full = torch.zeros((P, ng), dtype=C128, device=DEV)
    full[:, f.flat] = gam
    xbar = torch.fft.fftn(full.reshape((P,) + f.g), dim=(1, 2, 3)).reshape(P, ng).real
    rbar = torch.cholesky_solve(xbar.contiguous(), f.L)
    sbar = -rbar @ f.xi.T
    rbar[:, f.p] += sbar
    Y2 = 2.0 * rbar * f.B.conj()
    T1, T2 = Y2 @ U.T, U[:, f.p].conj() @ Y2
    g1 = (Uv.reshape(nk, nv, ng) @ T2.reshape(nk, no, ng).transpose(1, 2)).conj()
    g2 = Uv[:, f.p].conj().reshape(nk, nv, P) @ T1.reshape(P, nk, no).permute(1, 0, 2)
    return [ge + g1 + g2, ge, ex]
