"""The work that users of this library have it do, as measurable cases.

A Chebyshev-filtered subspace iteration calls the library three times per
self-consistency step: the Rayleigh-Ritz projection Hp = Psi^T (H Psi)
(Context.project), the density matrix D = f(Hp) with its band energy
(Context.solve, or Context.solve_batch for the k-points and spin channels of
one step), and the rotation Psi D (Context.rotate).  Context.gershgorin gives
spectral bounds alone.  Everything runs on device buffers through one Context
that the program keeps; a pass is one call.

Inputs are made on the GPU from the seed: Hp = Q diag(lambda) Q with
Q from a QR factorisation up to n = 1024 and Q = I - 2 V V^T (V n x 64
orthonormal) above, so D = Q f(lambda) Q^T is known exactly.
"""
import math
import random

import numpy as np
import torch

import paper_2301_04642_gb300 as fe

DEV = "cuda:0"
METHODS = {"auto": fe.FE_METHOD_AUTO, "asp2": fe.FE_METHOD_ASP2, "trfoe": fe.FE_METHOD_TRFOE}

_context = None


def _ctx():
    """The program's one library context."""
    global _context
    if _context is None:
        _context = fe.Context(device=0)
    return _context


# --------------------------------------------------------------------- cases
def listed():
    return [
        # the plain FP64 schedule on a small gapped Hp at a tight tolerance:
        # the reference run a user checks the fast schedules against
        dict(name="solve_fp64_n256", kind="solve", n=256, ne=200, lo=-2.0, hi=0.6, gap=0.1, kT=0.0, tol=1e-10,
             precision="fp64", method="auto", pad=0),
        # one small system in an interactive loop: the latency of a call
        dict(name="solve_n384", kind="solve", n=384, ne=300, lo=-2.0, hi=0.6, gap=0.1, kT=0.0, tol=0.0,
             precision="mixed", method="auto", pad=0),
        # a mid-size system after the first self-consistency step: HOMO / LUMO
        # estimates of the step before accelerate the expansion
        dict(name="asp2_n1250", kind="solve", n=1250, ne=1063, lo=-3.0, hi=1.0, gap=0.02, kT=0.0, tol=0.0,
             precision="mixed", method="asp2", pad=0),
        # the ordinary gapped solve
        dict(name="solve_n4096", kind="solve", n=4096, ne=3500, lo=-3.0, hi=1.0, gap=0.02, kT=0.0, tol=0.0,
             precision="mixed", method="auto", pad=0),
        # a small metal, odd n: Fermi-Dirac occupations
        dict(name="fermi_n517", kind="solve", n=517, ne=440, lo=-2.0, hi=1.0, gap=0.0, kT=0.01, tol=0.0,
             precision="mixed", method="auto", pad=0),
        # the largest: the finite-temperature workload of the benchmark
        dict(name="fermi_n16384", kind="solve", n=16384, ne=14000, lo=-2.0, hi=1.0, gap=0.0, kT=0.003, tol=0.0,
             precision="mixed", method="auto", pad=0),
        # k-points and spin channels of one step: a ragged batch in one call
        dict(name="batch_24", kind="batch", count=24, nmin=512, nmax=6144, mix=2000),
        # Rayleigh-Ritz projection: a large grid, and a small odd one with a
        # padded leading dimension
        dict(name="project_n4096", kind="project", m=131072, n=4096, pad=0),
        dict(name="project_n517", kind="project", m=9001, n=517, pad=3),
        # subspace rotation: a large grid, and a small one
        dict(name="rotate_n4096", kind="rotate", m=131072, n=4096, pad=0),
        dict(name="rotate_n300", kind="rotate", m=20000, n=300, pad=4),
        # spectral bounds alone
        dict(name="gershgorin_n8192", kind="gershgorin", n=8192, pad=0),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["solve", "solve", "asp2", "fp64", "fermi", "fermi", "trfoe", "batch", "project", "rotate",
                       "gershgorin"])
    pad = rng.choice([0, 0, 0, 1, 6])
    fill = rng.uniform(0.5, 0.92)
    if kind in ("solve", "asp2", "fp64"):
        n = _log(rng, *{"solve": (128, 8192), "asp2": (256, 4096), "fp64": (64, 1024)}[kind])
        return dict(kind="solve", n=n, ne=int(round(fill * n)), lo=-3.0, hi=1.0, gap=round(0.01 * 10 ** rng.random(), 4),
                    kT=0.0, tol=0.0, precision="fp64" if kind == "fp64" else "mixed",
                    method="asp2" if kind == "asp2" else "auto", pad=pad)
    if kind in ("fermi", "trfoe"):
        n = _log(rng, 128, 8192 if kind == "fermi" else 4096)
        return dict(kind="solve", n=n, ne=int(round(fill * n)), lo=-2.0, hi=1.0, gap=0.0,
                    kT=round(0.001 * 20 ** rng.random(), 5), tol=0.0, precision="mixed",
                    method="trfoe" if kind == "trfoe" else "auto", pad=pad)
    if kind == "batch":
        nmin = _log(rng, 128, 1024)
        return dict(kind="batch", count=rng.randint(4, 24), nmin=nmin, nmax=min(6144, _log(rng, 2, 12) * nmin),
                    mix=rng.randrange(10000))
    if kind == "gershgorin":
        return dict(kind=kind, n=_log(rng, 512, 16384), pad=pad)
    n = _log(rng, 128, 4096)
    return dict(kind=kind, m=_log(rng, max(n, 4096), 131072), n=n, pad=pad)


# -------------------------------------------------------------------- inputs
def _gen(seed):
    return torch.Generator(device=DEV).manual_seed(int(seed) * 7919 + 13)


def _rand(g, *shape):
    return torch.rand(*shape, generator=g, device=DEV, dtype=torch.float64)


def _randn(g, *shape):
    return torch.randn(*shape, generator=g, device=DEV, dtype=torch.float32).double()


def _padded(rows, cols, pad):
    """rows x cols with leading dimension cols + pad."""
    return torch.zeros(rows, cols + pad, device=DEV, dtype=torch.float64)[:, :cols]


def _levels(c, g):
    """The spectrum: two bands with a gap at 0 at zero temperature, the
    semicircle density on [lo, hi] at finite temperature; ascending."""
    n, ne = c["n"], c["ne"]
    if c["kT"] > 0.0:
        u = _rand(g, 2, n)
        x = torch.sqrt(u[0]) * torch.cos(2.0 * math.pi * u[1])
        return torch.sort(0.5 * (c["lo"] + c["hi"]) + 0.5 * (c["hi"] - c["lo"]) * x).values
    h = 0.5 * c["gap"]
    u = _rand(g, n)
    occ = torch.sort(c["lo"] + (-h - c["lo"]) * u[:ne]).values
    emp = torch.sort(h + (c["hi"] - h) * u[ne:]).values
    occ[-1:], emp[:1] = -h, h
    return torch.cat([occ, emp])


def _basis(n, g):
    """A function d -> Q diag(d) Q^T of a random orthogonal Q."""
    if n <= 1024:
        q = torch.linalg.qr(_randn(g, n, n)).Q
        return lambda d: (q * d) @ q.T
    v = torch.linalg.qr(_randn(g, n, 64)).Q

    def conjugate(d):
        # (I - 2 V V^T) diag(d) (I - 2 V V^T)
        w = v * d[:, None]
        h = torch.addmm(torch.diag(d), v, (w - v @ (v.T @ w)).T, alpha=-2.0)
        return h.addmm_(w - v @ (v.T @ w), v.T, alpha=-2.0)
    return conjugate


def _occupations(lam, ne, kT):
    """Step or Fermi-Dirac occupations of the levels in FP64, and mu."""
    lam = lam.cpu().numpy()
    if kT == 0.0:
        return (np.arange(lam.size) < ne).astype(np.float64), 0.0
    a, b = lam[0] - 50.0 * kT, lam[-1] + 50.0 * kT
    for _ in range(200):
        mu = 0.5 * (a + b)
        f = 0.5 * (1.0 - np.tanh((lam - mu) / (2.0 * kT)))
        a, b = (mu, b) if f.sum() < ne else (a, mu)
    return f, mu


def _members(c):
    """The solves of a batch: log-spread sizes, gaps and fillings."""
    r = random.Random(c["mix"])
    out = []
    for _ in range(c["count"]):
        n = _log(r, c["nmin"], c["nmax"])
        out.append(dict(n=n, ne=int(round(0.85 * n)), lo=-3.0, hi=1.0, gap=0.01 + 0.09 * r.random(), kT=0.0, pad=0))
    return out


def _hamiltonian(c, g):
    """Hp, its levels and the conjugation by its eigenvectors."""
    lam = _levels(c, g)
    q = _basis(c["n"], g)
    h = q(lam)
    out = _padded(c["n"], c["n"], c["pad"])
    torch.add(0.5 * h, h.T, alpha=0.5, out=out) if c["pad"] == 0 else out.copy_(0.5 * (h + h.T))
    return out, lam, q


def _block(c, g):
    """Psi: m x n filtered vectors, nearly orthonormal."""
    p = _padded(c["m"], c["n"], c["pad"])
    return p.copy_(_randn(g, c["m"], c["n"]).mul_(1.0 / math.sqrt(c["m"])))


def _problem(c, g):
    h, lam, _ = _hamiltonian(c, g)
    it = dict(H=h, ne=float(c["ne"]), kT=c["kT"], tol=c.get("tol", 0.0), D=_padded(c["n"], c["n"], c["pad"]),
              precision=c.get("precision", "mixed"), method=METHODS[c.get("method", "auto")])
    if c.get("method") == "asp2":
        # the step before knew the gap's edges to a tenth of its width
        it["homo"], it["lumo"] = -0.4 * c["gap"], 0.4 * c["gap"]
    return it


def _projection_inputs(c, g):
    psi = _block(c, g)
    # H Psi of nearly converged Ritz vectors: their levels times them plus a residual
    lam = _levels(dict(n=c["n"], ne=int(0.85 * c["n"]), lo=-3.0, hi=1.0, gap=0.02, kT=0.0), g)
    hpsi = _padded(c["m"], c["n"], c["pad"])
    hpsi.copy_(_randn(g, c["m"], c["n"]).mul_(0.05 / math.sqrt(c["m"])).addcmul_(psi, lam))
    return psi, hpsi


def _rotation_inputs(c, g):
    psi = _block(c, g)
    f = (torch.arange(c["n"], device=DEV) < int(0.85 * c["n"])).double()
    d = _basis(c["n"], g)(f)
    return psi, 0.5 * (d + d.T)


def prepare(case, seed):
    c, g = case, _gen(seed)
    s = dict(kind=c["kind"], ctx=_ctx())
    if c["kind"] == "solve":
        s["item"] = _problem(c, g)
    elif c["kind"] == "batch":
        s["items"] = [_problem(m, g) for m in _members(c)]
    elif c["kind"] == "project":
        s["psi"], s["hpsi"] = _projection_inputs(c, g)
        s["hp"] = _padded(c["n"], c["n"], 0)
    elif c["kind"] == "rotate":
        s["psi"], s["d"] = _rotation_inputs(c, g)
        s["out"] = _padded(c["m"], c["n"], c["pad"])
    else:
        s["h"] = _hamiltonian(dict(n=c["n"], ne=int(0.85 * c["n"]), lo=-3.0, hi=1.0, gap=0.02, kT=0.0, pad=c["pad"]), g)[0]
    return s


# ---------------------------------------------------------------------- pass
def _answer(it, r):
    out = dict(D=it["D"], e_band=r["e_band"], trace=r["trace"])
    if it["kT"] > 0.0:
        out["mu"] = r["mu"]
    return out


def run(s):
    ctx = s["ctx"]
    if s["kind"] == "solve":
        it = s["item"]
        return _answer(it, ctx.solve(**it))
    if s["kind"] == "batch":
        _, rs = ctx.solve_batch(s["items"])
        return dict(D=[it["D"] for it in s["items"]], e_band=np.array([r["e_band"] for r in rs]),
                    trace=np.array([r["trace"] for r in rs]))
    if s["kind"] == "project":
        ctx.project(s["psi"], s["hpsi"], s["hp"])
        return s["hp"]
    if s["kind"] == "rotate":
        ctx.rotate(s["psi"], s["d"], s["out"])
        return s["out"]
    return ctx.gershgorin(s["h"])


# ---------------------------------------------------------------- references
def _products(c):
    """Products of symmetric matrices an expansion needs: about two per
    halving of the gap (zero temperature) and one doubling with its inverse
    per halving of kT (finite temperature); the truncated expansion two per
    halving of kT."""
    w = c["hi"] - c["lo"]
    if c["kT"] > 0.0:
        return round((2 if c.get("method") == "trfoe" else 13) * math.log2(w / c["kT"]))
    p = 2.0 * math.log2(w / c["gap"]) + 18
    return round(0.6 * p if c.get("method") == "asp2" else p)


def work(case):
    c = case
    if c["kind"] in ("solve", "batch"):
        ms = [c] if c["kind"] == "solve" else _members(c)
        return {"bytes": float(sum(16 * m["n"] ** 2 for m in ms)),
                "flops": float(sum(_products(m) * m["n"] ** 2 * (m["n"] + 1) for m in ms))}
    if c["kind"] == "gershgorin":
        return {"bytes": 8.0 * c["n"] ** 2, "flops": 0.0}
    m, n = c["m"], c["n"]
    # the projection is symmetric: half the products
    return {"bytes": 8.0 * (2 * m * n + n * n), "flops": float(m * n * (n + 1) if c["kind"] == "project" else 2 * m * n * n)}


def _exact_solve(c, g):
    _, lam, q = _hamiltonian(c, g)
    f, mu = _occupations(lam, c["ne"], c["kT"])
    out = dict(D=q(torch.from_numpy(f).to(DEV)), e_band=float(np.sum(f * lam.cpu().numpy())), trace=float(c["ne"]))
    if c["kT"] > 0.0:
        out["mu"] = float(mu)
    return out


def exact(case, seed):
    c, g = case, _gen(seed)
    if c["kind"] == "solve":
        if c["method"] == "trfoe":
            return None  # a smeared step of its own, not Fermi-Dirac
        return _exact_solve(c, g)
    if c["kind"] == "batch":
        got = [_exact_solve(m, g) for m in _members(c)]
        return dict(D=[r["D"] for r in got], e_band=np.array([r["e_band"] for r in got]),
                    trace=np.array([r["trace"] for r in got]))
    if c["kind"] == "project":
        psi, hpsi = _projection_inputs(c, g)
        u = torch.triu(psi.T @ hpsi)  # the upper triangle counts, mirrored
        return u + torch.triu(u, 1).T
    if c["kind"] == "rotate":
        psi, d = _rotation_inputs(c, g)
        return psi @ d
    h = prepare(c, seed)["h"]
    d = torch.diagonal(h)
    r = h.abs().sum(1) - d.abs()
    return [float((d - r).min()), float((d + r).max()), float(d.sum()), 0.0]
