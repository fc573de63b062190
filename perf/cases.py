"""Performance cases of the grouped J/K framework: what its users run, through its public entry points.

A case is one of these kinds:
  build   a grouped build of m densities from a handle that exists (FockBuilder.build; integrals stored or direct)
  host    the same from and to page-locked host memory (FockBuilder.build_host)
  batch   several molecules of uneven size in one call (build_batch)
  create  a new geometry: the handle is made, used for one build and given back
  gvp     the GVP objective with its derivatives, one optimisation step of the method (FockBuilder.gvp_gradient)
  energy  the energy with its gradient (FockBuilder.energy_gradient)
  df      a build over density-fitted integrals
  thc     a build over hypercontracted integrals
Geometries and bases follow the repository's seeded recipes (workloads.py) at their densities of matter.
"""
import math

import numpy as np
import torch

from paper_2002_00322_gb300 import fock
from paper_2002_00322_gb300 import workloads as W

DEVICE = "cuda"
TOL = 1e-10
FIT_TOL, RIDGE = 1e-10, 1e-8
BATCH = [(40, 4), (44, 7), (48, 10), (52, 13), (56, 16), (60, 6), (64, 9), (68, 12),
         (72, 15), (76, 5), (80, 8), (84, 11), (88, 14), (92, 4), (96, 7), (100, 10)]


def listed():
    return [
        # a test-sized molecule, unscreened: launches and latency
        {"name": "tiny_n24_m4_fp64", "kind": "build", "n": 24, "m": 4, "precision": "fp64", "mode": "stored", "tol": 0.0, "shape": "cube"},
        # odd sizes, the nine densities of the method, called with host buffers by a program that keeps its matrices there
        {"name": "host_n77_m9_fp64", "kind": "host", "n": 77, "m": 9, "precision": "fp64", "mode": "stored", "tol": TOL, "shape": "cube"},
        # the headline workload in the default precision
        {"name": "stored_n200_m16_fp64", "kind": "build", "n": 200, "m": 16, "precision": "fp64", "mode": "stored", "tol": TOL, "shape": "cube"},
        # the same in the faster precisions
        {"name": "stored_n200_m16_fp32", "kind": "build", "n": 200, "m": 16, "precision": "fp32", "mode": "stored", "tol": TOL, "shape": "cube"},
        {"name": "stored_n200_m16_fp16x2", "kind": "build", "n": 200, "m": 16, "precision": "fp16x2", "mode": "stored", "tol": TOL, "shape": "cube"},
        # a larger molecule with many densities in one pass: throughput of the split store
        {"name": "stored_n400_m64_fp16x2", "kind": "build", "n": 400, "m": 64, "precision": "fp16x2", "mode": "stored", "tol": TOL, "shape": "cube"},
        # a long ribbon whose integrals are evaluated in every build
        {"name": "direct_n2000_m32_fp32", "kind": "build", "n": 2000, "m": 32, "precision": "fp32", "mode": "direct", "tol": TOL, "shape": "ribbon"},
        # s, p and d shells, the shape of a polarised basis
        {"name": "spd_n100_m16_fp64", "kind": "build", "n": 100, "m": 16, "precision": "fp64", "mode": "stored", "tol": TOL, "shape": "spd"},
        # one optimisation step: two builds of three densities and the matrix algebra around them
        {"name": "gvp_n200_fp64", "kind": "gvp", "n": 200, "m": 3, "precision": "fp64", "mode": "stored", "tol": TOL, "shape": "cube"},
        # density fitting, seven auxiliaries on each center
        {"name": "df_n200_m16_fp64", "kind": "df", "n": 200, "m": 16, "precision": "fp64", "mode": "df", "tol": TOL, "shape": "cube"},
        # sixteen small molecules of uneven size in one call, as a server's tick has them
        {"name": "batch_16x40to100_fp16x2", "kind": "batch", "n": 100, "m": 16, "precision": "fp16x2", "mode": "stored", "tol": TOL, "shape": "cube"},
        # every new geometry pays for its screening and integrals once
        {"name": "create_n120_m9_fp64", "kind": "create", "n": 120, "m": 9, "precision": "fp64", "mode": "stored", "tol": TOL, "shape": "cube"},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["build"] * 6 + ["host", "batch", "create", "gvp", "energy", "df", "thc"])
    c = {"kind": kind, "n": 0, "m": _log(rng, 1, 64), "precision": "fp64", "mode": "stored", "tol": TOL, "shape": "cube"}
    if kind in ("build", "host"):
        c["precision"] = rng.choice(["fp64", "fp64", "fp64", "f32x2", "fp32", "fp16x2", "bf16x2"])
        c["n"] = _log(rng, 9, 200 if c["precision"] in ("fp64", "f32x2") else 400)
        if kind == "build" and rng.random() < 0.2:
            # integral-direct over a ribbon of four rows
            c.update(mode="direct", shape="ribbon", precision=rng.choice(["fp64", "fp32", "fp16x2"]))
            c["n"] = 8 * _log(rng, 3, 20 if c["precision"] == "fp64" else 125)
        elif rng.random() < 0.2:
            c.update(shape="spd", n=10 * rng.randint(1, 10), precision=rng.choice(["fp64", "fp16x2"]))
    elif kind == "create":
        c["precision"] = rng.choice(["fp64", "fp32", "fp16x2"])
        c["n"] = _log(rng, 16, 160 if c["precision"] == "fp64" else 240)
    elif kind == "batch":
        c.update(precision=rng.choice(["fp16x2", "bf16x2"]), n=_log(rng, 40, 200), m=_log(rng, 4, 16))
    elif kind in ("gvp", "energy"):
        c.update(precision=rng.choice(["fp64", "fp64", "fp32", "fp16x2"]), n=_log(rng, 16, 200), m=3)
    elif kind == "df":
        c.update(precision=rng.choice(["fp64", "fp32"]), n=_log(rng, 16, 160), m=_log(rng, 1, 32), mode="df")
    else:
        c.update(precision=rng.choice(["fp64", "fp32"]), n=_log(rng, 16, 80), m=_log(rng, 1, 32), mode="thc")
    return c


# ------------------------------------------------------------------ inputs
def _rng(seed, salt):
    return np.random.Generator(np.random.PCG64([int(seed), salt]))


def _sizes(case):
    """(functions, densities) of a case's molecules: the batch scales the sixteen small molecules to its largest."""
    if case["kind"] != "batch":
        return [(case["n"], case["m"])]
    return [(max(2, round(n * case["n"] / 100)), max(1, round(m * case["m"] / 16))) for n, m in BATCH]


def _basis(n, shape, seed, salt=1):
    rng = _rng(seed, salt)
    if shape == "ribbon":
        return W.s_basis(rng, W.ribbon_centers(4, n // 8, 1.4), 2, 3)
    if shape == "spd":
        cen = W.cube_centers(rng, n // 10, 10.0 * (n / 1000.0) ** (1.0 / 3.0), 1.4)
        return W.spd_basis(rng, cen, nprim=2)
    ncen = (n + 1) // 2
    cen = W.cube_centers(rng, ncen, 10.0 * (ncen / 100.0) ** (1.0 / 3.0), 1.4 if ncen > 2 else 0.0)
    return W.s_basis(rng, cen, 2, 3).subset(np.arange(n))


def _densities(n, m, seed, salt=2):
    """The nine densities of the method, then transition densities (the recipe of workloads.esmf_densities, on the GPU)."""
    g = torch.Generator(DEVICE).manual_seed(int(seed) * 131 + salt)
    rnd = lambda *s: torch.randn(*s, generator=g, device=DEVICE, dtype=torch.float64)  # noqa: E731
    no = max(1, n // 5)
    V = torch.linalg.qr(rnd(n, n))[0].T.contiguous()
    Th, Ga = V[:no], V[no:]
    unit = lambda: (lambda x: x / x.norm())(rnd(no, n - no))  # noqa: E731
    s, mu = unit(), unit()
    M = rnd(n, n) / math.sqrt(n)
    Wt = (M - M.T).T @ V
    R, Phi = Wt[:no], Wt[no:]
    out = [Th.T @ Th, Th.T @ s @ Ga, Ga.T @ s.T @ s @ Ga - Th.T @ s @ s.T @ Th, R.T @ Th, R.T @ s @ Ga,
           Th.T @ mu @ Ga, Th.T @ s @ Phi, Th.T @ mu @ s.T @ Th, Phi.T @ s.T @ s @ Ga - R.T @ s @ s.T @ Th][:m]
    while len(out) < m:
        out.append(Th.T @ unit() @ Ga)
    return torch.stack(out)


def _orbital_state(basis, n, seed):
    """G, V, sigma, c0, n_occ of one wave function and the objective's omega, mu, chi."""
    st = W.esmf_state(_rng(seed, 3), basis, max(1, n // 5))
    t = lambda x: torch.from_numpy(np.ascontiguousarray(x)).to(DEVICE)  # noqa: E731
    return t(st.G), t(st.V), t(st.sigma), st.c0, st.nocc


OMEGA, MU, CHI = -1.5, 0.3, 0.6


def _builder(case, basis):
    if case["mode"] == "df":
        return fock.FockBuilder(basis, 0.0, "df", case["precision"], aux=W.even_tempered_aux(basis))
    if case["mode"] == "thc":
        return fock.FockBuilder(basis, FIT_TOL, "thc", case["precision"], grid=W.thc_grid(basis, corner=0), ridge=RIDGE)
    return fock.FockBuilder(basis, case["tol"], case["mode"], case["precision"])


def prepare(case, seed):
    kind = case["kind"]
    sizes = _sizes(case)
    bases = [_basis(n, case["shape"], seed, 1 + 10 * i) for i, (n, _) in enumerate(sizes)]
    st = {"case": case, "basis": bases[0]}
    if kind != "create":
        st["builders"] = [_builder(case, b) for b in bases]
    if kind in ("gvp", "energy"):
        st["state"] = _orbital_state(bases[0], case["n"], seed)
    else:
        st["D"] = [_densities(n, m, seed, 2 + 10 * i) for i, (n, m) in enumerate(sizes)]
    if kind == "host":
        pin = lambda x: torch.empty(x.shape, dtype=x.dtype, pin_memory=True)  # noqa: E731
        D = st["D"][0]
        st["host"] = [pin(D).copy_(D), pin(D), pin(D), torch.empty(len(D), dtype=torch.float64, pin_memory=True)]
    return st


# -------------------------------------------------------------------- a pass
def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "create":
        with _builder(case, state["basis"]) as fb:
            J, K, _, t = fb.build(state["D"][0])
        return {"J": J, "K": K, "traces": t}
    fb = state["builders"][0]
    if kind == "host":
        D, J, K, t = state["host"]
        fb.build_host(D, J, K, t)
        return {"J": J, "K": K, "traces": t}
    if kind == "batch":
        return [{"J": J, "K": K} for J, K in fock.build_batch(state["builders"], state["D"])]
    if kind == "gvp":
        G, V, s, c0, no = state["state"]
        scal, ds, dX = fb.gvp_gradient(G, V, s, c0, no, OMEGA, MU, CHI)
        return {"scalars": scal, "dsigma": ds, "dX": dX}
    if kind == "energy":
        G, V, s, c0, no = state["state"]
        scal, ds, dV = fb.energy_gradient(G, V, s, c0, no)
        return {"scalars": scal, "dsigma": ds, "dV": dV}
    J, K, _, t = fb.build(state["D"][0])
    return {"J": J, "K": K, "traces": t}


# ---------------------------------------------------- plain 64-bit evaluation
def _weights(basis):
    """Per function the exponents and the weights of its raw Gaussians, normalised (s functions)."""
    off = np.concatenate([[0], np.cumsum(basis.nprim)])
    a = np.stack([basis.exps[off[i]:off[i + 1]] for i in range(basis.n)])
    c = np.stack([basis.coefs[off[i]:off[i + 1]] for i in range(basis.n)])
    ov = (2.0 * np.sqrt(a[:, :, None] * a[:, None, :]) / (a[:, :, None] + a[:, None, :])) ** 1.5
    c = c / np.sqrt(np.einsum("ik,ikl,il->i", c, ov, c))[:, None]
    t = lambda x: torch.from_numpy(np.ascontiguousarray(x)).to(DEVICE)  # noqa: E731
    return t(a), t(c * (2.0 * a / math.pi) ** 0.75), t(basis.center)


def _pairs(basis):
    """Primitive pairs of the function pairs p >= q: exponent sums, product centers and weights, and the pairs' index table."""
    a, w, cen = _weights(basis)
    n = basis.n
    p, q = torch.tril_indices(n, n, device=DEVICE)
    e = a[p][:, :, None] + a[q][:, None, :]
    mu = a[p][:, :, None] * a[q][:, None, :] / e
    k = w[p][:, :, None] * w[q][:, None, :] * torch.exp(-mu * ((cen[p] - cen[q]) ** 2).sum(1)[:, None, None])
    P = (a[p][:, :, None, None] * cen[p][:, None, None] + a[q][:, None, :, None] * cen[q][:, None, None]) / e[..., None]
    idx = torch.empty(n, n, dtype=torch.long, device=DEVICE)
    idx[p, q] = idx[q, p] = torch.arange(len(p), device=DEVICE)
    f = lambda x: x.reshape(len(p), -1)  # noqa: E731
    return f(e), P.reshape(len(p), -1, 3), f(k), idx


def _boys(T):
    r = torch.sqrt(T.clamp_min(1e-6))
    big = 0.5 * math.sqrt(math.pi) * torch.erf(r) / r
    return torch.where(T < 1e-6, 1.0 - T / 3.0 + T * T / 10.0, big)


def _eri(x, y):
    """Contracted (x|y) of two lists of charge distributions (exponents, centers, weights; the last axis runs over primitives), broadcast."""
    e, P, k = x[0][..., :, None], x[1][..., :, None, :], x[2][..., :, None]
    f, Q, l = y[0][..., None, :], y[1][..., None, :, :], y[2][..., None, :]
    r2 = ((P - Q) ** 2).sum(-1)
    return (k * l * 2.0 * math.pi ** 2.5 / (e * f * torch.sqrt(e + f)) * _boys(e * f / (e + f) * r2)).sum((-1, -2))


def _integrals(basis, tol):
    """All (pq|rs) over pairs p >= q, zero where Q_pq Q_rs < tol."""
    e, P, k, idx = _pairs(basis)
    n = len(e)
    M = torch.empty(n, n, dtype=torch.float64, device=DEVICE)
    step = max(1, (1 << 25) // (n * e.shape[1] ** 2))
    for i in range(0, n, step):
        j = min(n, i + step)
        b = _eri((e[i:j, None], P[i:j, None], k[i:j, None]), (e[None, :j], P[None, :j], k[None, :j]))
        M[i:j, :j] = b
        M[:j, i:j] = b.T
    Q = torch.sqrt(M.diagonal().clamp_min(0.0))
    return M.mul_(Q[:, None] * Q[None, :] >= tol), idx


def _jk(M, idx, D):
    m, n = len(D), len(idx)
    p, q = torch.tril_indices(n, n, device=DEVICE)
    d = torch.where(p == q, D[:, p, q], D[:, p, q] + D[:, q, p])
    J = (d @ M)[:, idx]
    K = torch.empty_like(J)
    for i in range(n):
        T = M[idx[i]][:, idx.reshape(-1)].reshape(n, n, n)                  # [r][q][s] = (pr|qs)
        K[:, i] = D.reshape(m, -1) @ T.transpose(0, 1).reshape(n, -1).T
    return J, K


class _Fock(torch.autograd.Function):
    """F[D] = 2 J[D] - K[D]: linear and its own adjoint."""

    @staticmethod
    def forward(ctx, D, M, idx):
        ctx.of = M, idx
        J, K = _jk(M, idx, D[None])
        return 2.0 * J[0] - K[0]

    @staticmethod
    def backward(ctx, g):
        return _Fock.apply(g, *ctx.of), None, None


def _esmf_energy(G, V, s, c0, no, M, idx):
    Th, Ga = V[:no], V[no:]
    norm = c0 * c0 + 2.0 * (s * s).sum()
    P, T = Th.T @ Th, Th.T @ s @ Ga
    A = Ga.T @ s.T @ s @ Ga - Th.T @ s @ s.T @ Th
    FP, FT = _Fock.apply(P, M, idx), _Fock.apply(T, M, idx)
    e1 = 2.0 * norm * (G * P).sum() + 4.0 * c0 * (G * T).sum() + 2.0 * (G * A).sum()
    return (e1 + norm * (FP * P).sum() + 4.0 * c0 * (FP * T).sum() + 2.0 * (FP * A).sum() + 2.0 * (FT * T).sum()) / norm


def _exact_state(case, basis, seed):
    M, idx = _integrals(basis, case["tol"])
    G, V, s, c0, no = _orbital_state(basis, case["n"], seed)
    c0 = torch.tensor(c0, dtype=torch.float64, device=DEVICE, requires_grad=True)
    s.requires_grad_()
    if case["kind"] == "energy":
        V.requires_grad_()
        E = _esmf_energy(G, V, s, c0, no, M, idx)
        dc, ds, dV = torch.autograd.grad(E, (c0, s, V))
        return {"scalars": torch.stack([E.detach(), dc]), "dsigma": ds, "dV": dV}
    L = torch.zeros_like(V).requires_grad_()
    X = L.tril(-1) - L.tril(-1).T
    XV = X @ V
    E = _esmf_energy(G, V + XV + 0.5 * X @ XV, s, c0, no, M, idx)           # exp(X) V to the order that second derivatives see
    g = torch.autograd.grad(E, (c0, s, L), create_graph=True)
    g2 = sum((x * x).sum() for x in g)
    obj = CHI * (MU * (OMEGA - E) ** 2 + (1.0 - MU) * g2) + (1.0 - CHI) * E
    dc, ds, dL = torch.autograd.grad(obj, (c0, s, L))
    return {"scalars": torch.stack([obj.detach(), E.detach(), g2.detach(), dc]), "dsigma": ds, "dX": dL.tril(-1) - dL.tril(-1).T}


def _exact_df(basis, D):
    e, P, k, idx = _pairs(basis)
    cen, ex = W.even_tempered_aux(basis)
    t = lambda x: torch.from_numpy(np.ascontiguousarray(x)).to(DEVICE)  # noqa: E731
    aux = (t(ex)[:, None], t(cen)[:, None], torch.ones(len(ex), 1, dtype=torch.float64, device=DEVICE))
    T = torch.cat([_eri((e[i:i + 256, None], P[i:i + 256, None], k[i:i + 256, None]), tuple(x[None] for x in aux))
                   for i in range(0, len(e), 256)])
    V = _eri(tuple(x[:, None] for x in aux), tuple(x[None] for x in aux))
    B = torch.linalg.solve_triangular(torch.linalg.cholesky(V), T.T, upper=False)[:, idx]    # [P][p][q]
    J = torch.einsum("xpq,mx->mpq", B, torch.einsum("xrs,mrs->mx", B, D))
    K = torch.stack([torch.einsum("xps,xqs->pq", B @ d, B) for d in D])
    return J, K


def exact(case, seed):
    """Plain torch in 64 bits over all integrals. None above about 220 functions and for p and d functions, whose plain evaluation takes
    far over 20 seconds, and for hypercontraction, whose fit amplifies rounding by its conditioning (about 1 / ridge)."""
    sizes = _sizes(case)
    if case["shape"] == "spd" or case["kind"] == "thc" or max(n for n, _ in sizes) > 220:
        return None
    if case["kind"] == "batch" and case["n"] > 130:
        return None
    got = []
    for i, (n, m) in enumerate(sizes):
        basis = _basis(n, case["shape"], seed, 1 + 10 * i)
        if case["kind"] in ("gvp", "energy"):
            return _exact_state(case, basis, seed)
        D = _densities(n, m, seed, 2 + 10 * i)
        J, K = _exact_df(basis, D) if case["kind"] == "df" else _jk(*_integrals(basis, case["tol"]), D)
        got.append({"J": J, "K": K, "traces": (D * (2.0 * J - K)).sum((1, 2))})
    if case["kind"] == "batch":
        return [{"J": x["J"], "K": x["K"]} for x in got]
    return got[0]


# ---------------------------------------------------------------------- work
def _kept(case, n, salt):
    """Unique quartets that pass the Schwarz test, for one geometry of the case."""
    if case["tol"] == 0.0:
        k = n * (n + 1) // 2
        return k * (k + 1) // 2
    if case["shape"] == "spd":
        k = n * (n + 1) // 2
        return 0.96 * k * (k + 1) / 2
    e, P, k, _ = _pairs(_basis(n, case["shape"], 7, salt))
    rows = [tuple(t[i:i + 4096] for t in (e, P, k)) for i in range(0, len(e), 4096)]
    Q = torch.cat([_eri(x, x) for x in rows]).clamp_min(0.0).sqrt()
    Q = Q[Q > 0].sort().values
    ordered = (len(Q) - torch.searchsorted(Q, case["tol"] / Q)).sum()
    own = (Q * Q >= case["tol"]).sum()
    return int((ordered + own) // 2)


def work(case):
    """Each kept integral read once (or evaluated once), densities read and J, K written once; per kept unique quartet and density eight
    exchange and two Coulomb multiply-adds. Fitted builds: the contractions over their factors."""
    by, fl = 0.0, 0.0
    for i, (n, m) in enumerate(_sizes(case)):
        by += 3.0 * m * n * n * 8
        es = 8 if case["precision"] in ("fp64", "f32x2") else 4
        if case["kind"] in ("df", "thc"):
            cen = len(np.unique(_basis(n, case["shape"], 7).center, axis=0))
            if case["kind"] == "df":
                x = 7 * cen
                by += x * n * n * es
                fl += 4.0 * x * n * n * m + 4.0 * x * n ** 3 * m
            else:
                x = 13 * cen
                by += (x * n + x * x) * es
                fl += (6.0 * x * n * n + 4.0 * x * x * n + 2.0 * x * x) * m
            continue
        kept = _kept(case, n, 1 + 10 * i)
        passes = 2 if case["kind"] == "gvp" else 1
        by += passes * kept * es if case["mode"] == "stored" else 0.0
        fl += passes * 20.0 * m * kept
        if case["mode"] == "direct" or case["kind"] == "create":
            fl += 81.0 * 25.0 * kept
        if case["kind"] in ("gvp", "energy"):
            fl += passes * 14 * 2.0 * n ** 3
    return {"bytes": by, "flops": fl}
