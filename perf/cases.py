"""The work that users of the band-step library have it do, as cases that can be timed: band
steps of numerical-atomic-orbital cells from a few dozen to two thousand basis functions, their
eigenvalue-only and eigenvector forms, the mixed-precision form, a burst of serving requests and
the batched complex product, each through the public binding.

The cells are the repository's synthetic ones (Gaussian orbitals of heavy 13-orbital and light
8-orbital sites at random positions), generated here on the GPU so that new inputs are quick.

Outputs are quantities that do not depend on the free phase of an eigenvector: eigenvalues,
occupations, the Fermi level, the density matrices.  The one case that returns eigenvectors gives
them the usual convention of programs that store them (largest component real and positive).
"""
import math

import numpy as np
import torch

from paper_1402_4247_gb300 import nao, synth

DEV = "cuda:0"
HARTREE_EV = synth.HARTREE_EV


# --------------------------------------------------------------------------- the cases
def _step(name, heavy, light, kgrid, nspin, **more):
    """A band step: kgrid "4x4x4" (Monkhorst-Pack), nb eigenvector columns (0: all), edm: the
    energy density matrix too, images: cells out to that radius, eta: the overlap's
    regularisation exponents, dup: every dup-th orbital repeats its neighbour (0: none).
    kT is a smearing width (Hartree) that keeps the Fermi level of these sparse synthetic
    spectra well determined: inside a wide gap N(mu) is flat and any mu in it is as good."""
    case = dict(name=name, kind="step", heavy=heavy, light=light, kgrid=kgrid, nspin=nspin, images=1, nb=0,
                edm=False, kT=0.02, eta_lo=-3.0, eta_hi=-1.0, dup=0)
    case.update(more)
    return case


def listed():
    return [
        # a molecule-sized cell on a small k grid, the smallest step in use (the smoke test's
        # sizes): launches and latency count
        _step("step_n64_k4", 0, 8, "2x2x1", 1, kT=0.2),
        # a small two-spin cell with odd order and both density matrices (forces are wanted)
        _step("step_n129_k6_edm", 5, 8, "3x2x1", 2, edm=True, kT=0.05),
        # an ordinary cell in a self-consistency loop, eigenvectors of the occupied bands only
        _step("step_n305_k27_nb", 13, 17, "3x3x3", 1, nb=122),
        # the magnetite-shaped step: 128 problems, all eigenvectors
        _step("step_n568_k64_s2", 24, 32, "4x4x4", 2, images=2),
        # the same cell at a single k-point: a large supercell's self-consistency step
        _step("step_n568_k1_s2", 24, 32, "1x1x1", 2),
        # an overcomplete basis: one orbital in 50 repeats another, so directions are cut and
        # the smallest kept overlap eigenvalues are ~1e-4.  (The generator's 1e-8 setting leaves
        # eigenvalues of FP64 methods uncertain by 1e-6 and cannot be compared.)
        _step("step_n600_k8_cut", 24, 36, "2x2x2", 1, dup=50, eta_lo=-4.0, eta_hi=-2.0),
        # a large basis at one k-point, lowest bands
        _step("step_n2000_k1_nb", 80, 120, "1x1x1", 1, nb=700),
        # band structure along a line: eigenvalues only
        dict(name="bands_n449_k40", kind="bands", heavy=21, light=22, nk=40, images=1, eta_lo=-3.0, eta_hi=-1.0,
             mixed=False),
        # the same in the mixed-precision mode on the magnetite-shaped cell
        dict(name="bands_n568_k24_mixed", kind="bands", heavy=24, light=32, nk=24, images=1, eta_lo=-3.0,
             eta_hi=-1.0, mixed=True),
        # all eigenvectors of a batch of pencils that the caller assembled
        dict(name="vectors_n211_p24", kind="vectors", heavy=11, light=8, nk=24, images=1, eta_lo=-3.0, eta_hi=-1.0),
        # a burst of small serving requests of mixed order, k-points and spin
        dict(name="serve_r8_n64_300", kind="serve", requests=8, n_lo=64, n_hi=300),
        # batched complex products of odd sizes (post-processing of eigenvectors)
        dict(name="zgemm_p24_301_257_420", kind="zgemm", nprob=24, M=301, N=257, K=420),
    ]


_GRIDS = ("1x1x1", "2x1x1", "2x2x1", "3x2x1", "2x2x2", "3x3x1", "3x2x2", "4x4x1", "3x3x2", "3x3x3", "4x4x2", "4x4x4")


def _log_uniform(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def _sites(rng, n):
    """Heavy and light sites of a cell of about n orbitals."""
    heavy = int(rng.uniform(0.2, 0.7) * n / 13)
    return heavy, max(1, (n - 13 * heavy) // 8)


def draw(rng):
    kind = rng.choice(("step", "step", "step", "step", "bands", "vectors", "serve", "zgemm"))
    budget = 0.8 * 128 * 568 ** 3  # problems x n^3 of the largest listed step
    if kind == "zgemm":
        while True:
            M, N, K = (int(_log_uniform(rng, 8, 1200)) for _ in range(3))
            p = int(_log_uniform(rng, 1, 128))
            if p * (M * N + N * K + M * K) * 16 < 2 << 30 and p * M * N * K < 2e10:
                return dict(kind="zgemm", nprob=p, M=M, N=N, K=K)
    if kind == "serve":
        lo = int(_log_uniform(rng, 40, 200))
        return dict(kind="serve", requests=rng.randint(2, 10), n_lo=lo, n_hi=int(lo * _log_uniform(rng, 1.0, 3.0)))
    n = int(_log_uniform(rng, 24, 1100))
    heavy, light = _sites(rng, n)
    n = 13 * heavy + 8 * light
    pmax = max(1, min(128, int(budget / n ** 3)))
    if kind == "bands" or kind == "vectors":
        nk = max(1, int(_log_uniform(rng, 1, min(pmax, 64) + 0.5)))
        c = dict(kind=kind, heavy=heavy, light=light, nk=nk, images=1, eta_lo=-3.0, eta_hi=-1.0)
        if kind == "bands":
            c["mixed"] = rng.random() < 0.4
        return c
    nspin = rng.choice((1, 2))
    grids = [g for g in _GRIDS if nspin * _nk(g) <= pmax] or ["1x1x1"]
    c = _step("", heavy, light, rng.choice(grids), nspin)
    del c["name"]
    if n < 200:
        c["kT"] = 0.2 if n < 100 else 0.05
    elif rng.random() < 0.4:
        c["nb"] = int(0.42 * n)
    c["edm"] = rng.random() < 0.3
    if n <= 600 and rng.random() < 0.3:
        c["images"] = 2
    if n >= 100 and rng.random() < 0.2:
        c.update(dup=50, eta_lo=-4.0, eta_hi=-2.0, nb=0)
    return c


# --------------------------------------------------------------------------- inputs
def _nk(grid):
    return math.prod(int(x) for x in grid.split("x"))


def _kline(nk):
    """A line through the Brillouin zone from its centre towards a corner."""
    t = np.linspace(0.0, 0.5, nk) if nk > 1 else np.zeros(1)
    return np.stack([t, 0.7 * t, 0.3 * t], axis=1), np.full(nk, 1.0 / nk)


def _positions(rng, natom, side):
    """Seeded positions at least 1.8 Angstrom apart (minimum image)."""
    pos = np.zeros((natom, 3))
    placed = 0
    while placed < natom:
        p = rng.uniform(0.0, side, size=3)
        d = pos[:placed] - p
        d -= side * np.round(d / side)
        if placed and np.min(np.einsum("ij,ij->i", d, d)) < 1.8 * 1.8:
            continue
        pos[placed] = p
        placed += 1
    return pos


def _cell(seed, heavy, light, images, nspin, eta_lo, eta_hi, dup=0):
    """HR [nspin][nR][n][n], SR [nR][n][n] (Hartree), R [nR][3] on the GPU: the model of
    synth.make_cell, evaluated with torch."""
    rng = np.random.Generator(np.random.PCG64(seed))
    natom = heavy + light
    side = 8.4 * (natom / 56.0) ** (1.0 / 3.0)
    if natom < 56:
        side = 8.4 * max(natom / 56.0, 0.15) ** (1.0 / 3.0) + 2.0
    pos = _positions(rng, natom, side)
    norb = np.array([13] * heavy + [8] * light)
    atom = np.repeat(np.arange(natom), norb)
    is_heavy = atom < heavy
    n = atom.size
    sig = np.where(is_heavy, rng.uniform(1.0, 1.8, n), rng.uniform(0.7, 1.2, n))
    eta = 10.0 ** rng.uniform(eta_lo, eta_hi, n)
    onsite = rng.normal(0.0, 3.0, n) / HARTREE_EV
    delta = np.where(is_heavy, rng.uniform(1.0, 3.0, n), 0.0) / HARTREE_EV
    src = np.arange(n)  # the orbital each one copies
    if dup:
        for t in range(dup - 1, n, dup):
            s = t - 1 if t > 0 and atom[t - 1] == atom[t] else t + 1
            if s < n and atom[s] == atom[t]:
                src[t] = s
    R = synth.image_cube(images)
    g = torch.Generator(device=DEV).manual_seed(seed)
    f64 = dict(dtype=torch.float64, device=DEV)
    t = 0.5 + 1.5 * torch.rand((n, n), generator=g, **f64)
    t = torch.triu(t) + torch.triu(t, 1).T
    c = torch.from_numpy(pos[atom]).to(DEV)
    s = torch.from_numpy(sig).to(DEV)
    s2 = s[:, None] ** 2 + s[None, :] ** 2
    pref = (2.0 * s[:, None] * s[None, :] / s2) ** 1.5
    dvec = c[:, None, :] - c[None, :, :]
    d0 = torch.from_numpy(eta).to(DEV)
    SR = torch.empty((R.shape[0], n, n), **f64)
    HR = torch.empty((nspin, R.shape[0], n, n), **f64)
    for ir in range(R.shape[0]):
        shift = torch.tensor(side * R[ir].astype(np.float64), device=DEV)
        gauss = torch.exp(-((dvec - shift) ** 2).sum(-1) / s2)
        SR[ir] = pref * gauss
        HR[0, ir] = -(t / HARTREE_EV) * gauss
    r0 = int(np.flatnonzero(~R.any(axis=1))[0])
    SR[r0] += torch.diag(d0)
    HR[0, r0] += torch.diag(torch.from_numpy(onsite).to(DEV))
    delta = torch.from_numpy(delta).to(DEV)
    if dup:
        k = torch.from_numpy(src).to(DEV)
        SR = SR[:, k][:, :, k].contiguous()
        HR[0] = HR[0][:, k][:, :, k]
        d0, delta = d0[k], delta[k]
    dinv = 1.0 / torch.sqrt(1.0 + d0)
    SR = SR * dinv[None, :, None] * dinv[None, None, :]
    if nspin == 2:
        HR[1] = HR[0]
        HR[1, r0] += torch.diag(delta)
    return HR, SR, torch.from_numpy(R).to(DEV)


def _step_inputs(seed, case, kpts, wk):
    nspin = case.get("nspin", 1)
    HR, SR, R = _cell(seed, case["heavy"], case["light"], case["images"], nspin, case["eta_lo"], case["eta_hi"],
                      case.get("dup", 0))
    n, nk = SR.shape[1], kpts.shape[0]
    return dict(HR=HR, SR=SR, R=R, k=torch.from_numpy(np.ascontiguousarray(kpts)).to(DEV),
                w=torch.from_numpy(wk).to(DEV), n=n, nk=nk, nspin=nspin, ne=2.0 * (n // 4),
                smap=torch.arange(nspin * nk, dtype=torch.int32, device=DEV) % nk)


def _serve_sizes(case):
    """(heavy, light, kgrid, nspin) of each request of a burst."""
    out = []
    q = case["requests"]
    for i in range(q):
        n = int(round(case["n_lo"] * (case["n_hi"] / case["n_lo"]) ** (i / max(1, q - 1))))
        heavy = int(0.4 * n / 13)
        out.append((heavy, max(1, (n - 13 * heavy) // 8), ("2x1x1", "1x1x1", "2x2x1", "2x2x2")[i % 4], 1 + i % 2))
    return out


_SERVE_KT = 0.2
_contexts = {}


def _context(serving=False):
    """The one library context that a program keeps (and one whose scheduler serves)."""
    if serving not in _contexts:
        c = _contexts[serving] = nao.Context(0)
        if serving:
            c.nao_serve_config(24 << 30, 64, 2)
    return _contexts[serving]


def _grid(text):
    return synth.monkhorst_pack(*(int(x) for x in text.split("x")))


def _zgemm_inputs(case, seed):
    g = torch.Generator(device=DEV).manual_seed(seed)
    shapes = ((case["nprob"], case["M"], case["K"]), (case["nprob"], case["K"], case["N"]))
    return [torch.randn(s, generator=g, dtype=torch.complex128, device=DEV) for s in shapes]


def prepare(case, seed):
    kind = case["kind"]
    if kind == "zgemm":
        A, B = _zgemm_inputs(case, seed)
        return dict(case=case, ctx=_context(), A=A, B=B)
    if kind == "serve":
        reqs = []
        for i, (heavy, light, grid, nspin) in enumerate(_serve_sizes(case)):
            c = dict(heavy=heavy, light=light, images=1, nspin=nspin, eta_lo=-3.0, eta_hi=-1.0)
            reqs.append(_step_inputs(seed * 64 + i, c, *_grid(grid)))
        return dict(case=case, ctx=_context(serving=True), reqs=reqs)
    kpts, wk = _grid(case["kgrid"]) if kind == "step" else _kline(case["nk"])
    s = _step_inputs(seed, case, kpts, wk)
    s.update(case=case, ctx=_context())
    if kind == "vectors":
        n = s["n"]
        s["Hk"] = s["ctx"].nao_bloch_sum(s["HR"], s["R"], s["k"]).reshape(-1, n, n)
        s["Sk"] = s["ctx"].nao_bloch_sum(s["SR"][None], s["R"], s["k"])[0]
    return s


# --------------------------------------------------------------------------- one pass
def _largest_positive(C):
    """Each eigenvector's free phase fixed: its largest component real and positive."""
    i = C.abs().argmax(dim=-2, keepdim=True)
    z = torch.gather(C, -2, i)
    return C * (z.conj() / z.abs().clamp_min(1e-300))


def run(state):
    case, ctx = state["case"], state["ctx"]
    kind = case["kind"]
    if kind == "zgemm":
        return ctx.nao_zgemm(state["A"], state["B"])
    if kind == "serve":
        ctx.nao_serve_pause(True)
        tickets = [ctx.nao_serve_submit(q["HR"], q["SR"], q["R"], q["k"], q["w"], q["ne"], _SERVE_KT)
                   for q in state["reqs"]]
        ctx.nao_serve_pause(False)
        out = []
        for t in tickets:
            r = ctx.serve_result_tensors(ctx.nao_serve_poll(t))
            out.append({key: r[key] for key in ("eps", "m", "status", "mu", "rho")})
            ctx.nao_serve_release(t)
        return out
    n = state["n"]
    if kind == "vectors":
        eps, C, m, status = ctx.nao_gen_eig(state["Hk"], state["Sk"])
        return dict(eps=eps, C=_largest_positive(C), m=m, status=status)
    Sk = ctx.nao_bloch_sum(state["SR"][None], state["R"], state["k"])[0]
    Hk = ctx.nao_bloch_sum(state["HR"], state["R"], state["k"]).reshape(-1, n, n)
    if kind == "bands":
        eps, _, m, status = ctx.nao_gen_eig(Hk, Sk, precision=nao.NAO_MIXED_BF16X3 if case["mixed"] else nao.NAO_FP64,
                                            want_vectors=False)
        return dict(eps=eps, m=m, status=status)
    eps, C, m, status = ctx.nao_gen_eig(Hk, Sk, s_of_prob=state["smap"], nb=case["nb"] or n)
    edm = torch.empty_like(state["HR"]) if case["edm"] else None
    mu, eband, f, rho, rstatus = ctx.nao_density_matrix(state["w"], state["k"], eps, C, m, state["ne"], case["kT"],
                                                        state["R"], state["nspin"], edm=edm)
    out = dict(eps=eps, m=m, status=status, mu=mu, eband=eband, f=f, rho=rho, rstatus=rstatus)
    if edm is not None:
        out["edm"] = edm
    return out


# --------------------------------------------------------------------------- the least work
def _eig_work(n, nk, nspin, nR, nb, vectors):
    """FP64 operations of one Hermitian-definite eigenproblem per (spin, k): Cholesky factor,
    reduction to standard form, tridiagonalization, back-transformations of nb vectors; the
    Bloch sums' lower triangles before it."""
    p = nspin * nk
    flops = nk * 4 / 3 * n ** 3 + p * (4 + 16 / 3) * n ** 3 + (nspin + 1) * nk * 2 * nR * n * n
    if vectors:
        flops += p * (8 + 4) * n * n * nb
    return flops, (nspin + 1) * nR * n * n * 8 + p * n * 8


def work(case):
    kind = case["kind"]
    if kind == "zgemm":
        p, M, N, K = case["nprob"], case["M"], case["N"], case["K"]
        return {"bytes": 16 * p * (M * K + K * N + M * N), "flops": 8 * p * M * N * K}
    if kind == "serve":
        total = {"bytes": 0, "flops": 0}
        for heavy, light, grid, nspin in _serve_sizes(case):
            w = work(dict(kind="step", heavy=heavy, light=light, kgrid=grid, nspin=nspin, images=1, nb=0, edm=False))
            total = {k: total[k] + w[k] for k in total}
        return total
    n = 13 * case["heavy"] + 8 * case["light"]
    nR = (2 * case["images"] + 1) ** 3
    if kind == "bands":
        flops, nbytes = _eig_work(n, case["nk"], 1, nR, 0, False)
        return {"bytes": nbytes, "flops": flops}
    if kind == "vectors":
        flops, _ = _eig_work(n, case["nk"], 1, 0, n, True)
        return {"bytes": case["nk"] * (3 * 16 * n * n + 8 * n), "flops": flops}
    nk, nspin = _nk(case["kgrid"]), case["nspin"]
    flops, nbytes = _eig_work(n, nk, nspin, nR, case["nb"] or n, True)
    mats = 2 if case["edm"] else 1
    # the density matrices: a quarter of the bands occupied, half of each Hermitian product
    flops += mats * nspin * nk * (4 * n * n * (n // 4) + 4 * nR * n * n)
    return {"bytes": nbytes + mats * nspin * nR * n * n * 8 + nspin * nk * n * 8, "flops": flops}


# --------------------------------------------------------------------------- in 64 bits
def _bloch(MR, R, k, sign=1.0):
    """sum_r exp(2 pi i k.R) M(R), exactly Hermitian from the lower triangle."""
    ph = torch.exp(2j * math.pi * sign * (k @ R.to(torch.float64).T))
    n = MR.shape[-1]
    M = (ph @ MR.reshape(MR.shape[0], n * n).to(torch.complex128)).reshape(-1, n, n)
    low = torch.tril(M, -1)
    return low + low.mH + torch.diag_embed(torch.diagonal(M, dim1=-2, dim2=-1).real).to(M.dtype)


def _orthogonaliser(S, cut=1e-10):
    """X with X^H S X = 1 over the overlap eigenvalues from the cutoff up."""
    s, U = torch.linalg.eigh(S)
    keep = s >= cut
    return U[:, keep] / torch.sqrt(s[keep])


def _pencil(H, S, X=None):
    X = _orthogonaliser(S) if X is None else X
    Hp = X.mH @ H @ X
    e, V = torch.linalg.eigh(0.5 * (Hp + Hp.mH))
    return e, X @ V


def _fermi(e, w, ne, kT, g):
    """mu, f, E_band for eigenvalues e [nspin][nk][n] (inf where there is none)."""
    w = w[None, :, None]
    lo, hi = float(e[torch.isfinite(e)].min()) - 40 * kT, float(e[torch.isfinite(e)].max()) + 40 * kT
    occ = lambda mu: 1.0 / (1.0 + torch.exp(((e - mu) / kT).clamp(max=700.0)))  # noqa: E731
    for _ in range(200):
        mid = 0.5 * (lo + hi)
        if mid <= lo or mid >= hi:
            break
        if g * float((w * occ(mid)).sum()) < ne:
            lo = mid
        else:
            hi = mid
    mu = 0.5 * (lo + hi)
    f = torch.where(torch.isfinite(e), occ(mu), torch.zeros_like(e))
    return mu, f, g * (w * f * torch.where(torch.isfinite(e), e, torch.zeros_like(e))).sum()


def _exact_step(s, kT, want_edm):
    n, nk, nspin = s["n"], s["nk"], s["nspin"]
    S = _bloch(s["SR"], s["R"], s["k"])
    eps = torch.full((nspin, nk, n), math.inf, dtype=torch.float64, device=DEV)
    C = torch.zeros((nspin, nk, n, n), dtype=torch.complex128, device=DEV)
    Xs = [_orthogonaliser(S[q]) for q in range(nk)]
    for sp in range(nspin):
        H = _bloch(s["HR"][sp], s["R"], s["k"])
        for q in range(nk):
            e, c = _pencil(H[q], S[q], Xs[q])
            eps[sp, q, :e.numel()] = e
            C[sp, q, :, :e.numel()] = c
    g = 2.0 if nspin == 1 else 1.0
    mu, f, eband = _fermi(eps, s["w"], s["ne"], kT, g)
    ph = torch.exp(-2j * math.pi * (s["R"].to(torch.float64) @ s["k"].T)) * (g * s["w"])[None, :]
    fin = torch.where(torch.isfinite(eps), eps, torch.zeros_like(eps))

    def density(weights):
        out = torch.empty((nspin, ph.shape[0], n, n), dtype=torch.float64, device=DEV)
        for sp in range(nspin):
            P = (C[sp] * weights[sp][:, None, :]) @ C[sp].mH
            out[sp] = (ph @ P.reshape(nk, n * n)).real.reshape(-1, n, n)
        return out

    res = dict(eps=eps.reshape(nspin * nk, n), mu=torch.tensor([mu], dtype=torch.float64), eband=eband.reshape(1),
               f=f.reshape(nspin * nk, n), rho=density(f))
    if want_edm:
        res["edm"] = density(f * fin)
    return res


def exact(case, seed):
    kind = case["kind"]
    if kind == "zgemm":
        A, B = _zgemm_inputs(case, seed)
        return A @ B
    if kind == "serve":
        out = []
        for i, (heavy, light, grid, nspin) in enumerate(_serve_sizes(case)):
            c = dict(heavy=heavy, light=light, images=1, nspin=nspin, eta_lo=-3.0, eta_hi=-1.0)
            r = _exact_step(_step_inputs(seed * 64 + i, c, *_grid(grid)), _SERVE_KT, False)
            out.append({k: r[k] for k in ("eps", "mu", "rho")})
        return out
    kpts, wk = _grid(case["kgrid"]) if kind == "step" else _kline(case["nk"])
    s = _step_inputs(seed, case, kpts, wk)
    if kind == "step":
        return _exact_step(s, case["kT"], case["edm"])
    S = _bloch(s["SR"], s["R"], s["k"])
    H = _bloch(s["HR"][0], s["R"], s["k"])
    eps, C = zip(*(_pencil(H[q], S[q]) for q in range(s["nk"])))
    if kind == "bands":
        return dict(eps=torch.stack(eps))
    return dict(eps=torch.stack(eps), C=_largest_positive(torch.stack(C)))
