"""The work that is timed: calls of the public entry points over the sizes they are used at.

Lattices, widths, masses, shift counts and rational approximations are those of this repository's
workloads and tests: 4^4 .. 24^4 links exp(i eps H), 1 .. 16 right-hand sides, the Remez coefficients
of ``rational_coeffs.json``.  The mixed-precision solves run to 1e-11, the tolerance of the
finite-difference check of the gradient, the FP64 ones to 1e-12 (molecular dynamics), 1e-13 or 1e-14
(heatbath and accept/reject): there the answers are determined well beyond the rounding of one layer.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_1808_01829_gb300 import functional as rhmc
from paper_1808_01829_gb300 import hmc
from paper_1808_01829_gb300.api import RhmcContext, block_multishift_cg_batch
from paper_1808_01829_gb300.remez import rational_approx

DEV = "cuda"
BETA = 5.12  # Wilson coupling of the paper's runs


def listed():
    return [
        # one application of the operator on the paper's lattice: inside a caller's own Krylov solver
        {"name": "operator 8^4 n4 fp64", "kind": "operator", "lx": 8, "ly": 8, "lz": 8, "lt": 8, "n": 4, "mass": 0.05,
         "precision": "fp64"},
        # residual checks of a mid-size ensemble with the double-float operator, extents all different
        {"name": "operator 16x12x10x20 n5 df64", "kind": "operator", "lx": 16, "ly": 12, "lz": 10, "lt": 20, "n": 5,
         "mass": 0.02, "precision": "df64"},
        # the same operator at the largest workload
        {"name": "operator 24^4 n16 fp64", "kind": "operator", "lx": 24, "ly": 24, "lz": 24, "lt": 24, "n": 16,
         "mass": 0.01, "precision": "fp64"},
        # the smallest solve of the workloads: latency of the coefficient steps and launches
        {"name": "solve 4^4 n2 fp64", "kind": "solve", "lx": 4, "ly": 4, "lz": 4, "lt": 4, "n": 2, "mass": 0.1,
         "eps": 0.3, "r": -0.125, "low": 1e-3, "shifts": 8, "tol": 1e-12, "precision": "fp64"},
        # FP64 molecular dynamics on the paper's lattice
        {"name": "solve 8^4 n4 fp64", "kind": "solve", "lx": 8, "ly": 8, "lz": 8, "lt": 8, "n": 4, "mass": 0.05,
         "eps": 0.5, "r": -0.0625, "low": 2e-3, "shifts": 12, "tol": 1e-12, "precision": "fp64"},
        # mixed-precision solve, the 16^3 x 32 workload
        {"name": "solve 16^3x32 n8 mixed", "kind": "solve", "lx": 16, "ly": 16, "lz": 16, "lt": 32, "n": 8,
         "mass": 0.02, "eps": 0.5, "r": -0.03125, "low": 1e-3, "shifts": 14, "tol": 1e-11, "precision": "mixed"},
        # the force evaluation of the largest workload: links staged, solve, force
        {"name": "force 24^4 n16 mixed", "kind": "force", "lx": 24, "ly": 24, "lz": 24, "lt": 24, "n": 16,
         "mass": 0.01, "eps": 0.5, "r": -0.015625, "low": 4e-4, "shifts": 16, "tol": 1e-11, "precision": "mixed"},
        # pseudofermion heatbath phi = A^(1/(8 n)) eta: the rational sum alone, no shifted solutions
        {"name": "heatbath 12^4 n4 fp64", "kind": "heatbath", "lx": 12, "ly": 12, "lz": 12, "lt": 12, "n": 4,
         "mass": 0.025, "eps": 0.5, "r": 0.03125, "low": 2e-3, "shifts": 12, "tol": 1e-14},
        # the action as a differentiable function: forward and backward, gradients of U and Phi
        {"name": "action+grad 12^4 n4 mixed", "kind": "action", "lx": 12, "ly": 12, "lz": 12, "lt": 12, "n": 4,
         "mass": 0.025, "eps": 0.5, "r": -0.0625, "low": 2e-3, "shifts": 12, "tol": 1e-11, "precision": "mixed"},
        # three uneven ensembles solved at once (the smaller members of the batched workload)
        {"name": "batch 8^4 12^4 16^4 mixed", "kind": "batch", "first": 8, "members": 3, "mass": 0.025, "eps": 0.5,
         "low": 2e-3, "shifts": 12, "tol": 1e-11, "precision": "mixed"},
        # pure-gauge molecular dynamics: gauge-force kicks and link updates
        {"name": "gauge md 16^3x32", "kind": "md", "lx": 16, "ly": 16, "lz": 16, "lt": 32, "n": 0, "mass": 0.02,
         "eps": 0.5, "tau": 0.2, "steps": 2, "inner": 3, "tol": 1e-11, "precision": "mixed"},
        # a short RHMC trajectory on the paper's lattice: heatbath, action, MD, accept/reject
        {"name": "trajectory 8^4 n4", "kind": "trajectory", "lx": 8, "ly": 8, "lz": 8, "lt": 8, "n": 4,
         "mass": 0.025, "eps": 0.5, "tau": 0.2, "steps": 2, "inner": 3, "tol": 1e-11, "precision": "mixed"},
    ]


# (n, exponent, lower end, poles) of the approximations at hand: force -1/(4n), heatbath +1/(8n)
FORCE = [(1, -0.25, 2e-3, 12), (1, -0.25, 4e-4, 16), (2, -0.125, 1e-3, 8), (2, -0.125, 2e-3, 12), (3, -1 / 12, 1e-3, 5),
         (4, -0.0625, 2e-3, 12), (4, -0.0625, 4e-4, 16), (5, -0.05, 1e-3, 6), (6, -1 / 24, 1e-3, 5),
         (8, -0.03125, 1e-3, 14), (8, -0.03125, 2e-3, 12), (12, -1 / 48, 2e-3, 12), (16, -0.015625, 2e-3, 12),
         (16, -0.015625, 4e-4, 16)]
HEATBATH = [(1, 0.125, 2e-3, 12), (2, 0.0625, 2e-3, 12), (2, 0.0625, 1e-3, 8), (4, 0.03125, 2e-3, 12),
            (8, 0.015625, 2e-3, 12), (16, 0.0078125, 2e-3, 12), (16, 0.0078125, 4e-4, 24)]


def _extents(rng, low, high):
    """Four even extents with low <= volume <= high, the volume about log-uniform."""
    want = math.exp(rng.uniform(math.log(low), math.log(high)))
    while True:
        side = want ** 0.25
        d = [2 * max(1, round(side * rng.uniform(0.7, 1.4) / 2)) for _ in range(4)]
        if low <= d[0] * d[1] * d[2] * d[3] <= high and min(d) >= 4:
            return {"lx": d[0], "ly": d[1], "lz": d[2], "lt": d[3]}


def _mass(rng, low):
    """A mass whose 4 m^2 lies inside the approximation's interval."""
    m0 = math.sqrt(low) / 2
    return round(m0 * rng.uniform(1.05, 3.0), 4)


def draw(rng):
    kind = rng.choice(["operator", "operator", "solve", "solve", "force", "heatbath", "action", "batch", "md",
                       "trajectory"])
    c = {"kind": kind}
    if kind == "operator":
        c |= _extents(rng, 256, 331776)
        c |= {"n": rng.randint(1, 16), "mass": round(rng.uniform(0.01, 0.1), 4),
              "precision": rng.choice(["fp64", "fp64", "df64"])}
        return c
    if kind == "batch":
        c |= {"first": rng.choice([4, 6, 8, 10]), "members": rng.randint(2, 3), "mass": _mass(rng, 2e-3), "eps": 0.5,
              "low": 2e-3, "shifts": 12, "tol": 1e-11, "precision": "mixed"}
        return c
    c["eps"] = rng.choice([0.3, 0.5])
    if kind == "md":
        c |= _extents(rng, 256, 131072)
        c |= {"n": 0, "mass": 0.02, "tau": round(rng.uniform(0.05, 0.3), 3), "steps": rng.randint(1, 3),
              "inner": rng.randint(1, 3), "tol": 1e-11, "precision": "mixed"}
        return c
    if kind == "trajectory":
        c |= _extents(rng, 256, 6000)
        c |= {"n": rng.choice([1, 2, 4, 8]), "mass": _mass(rng, 2e-3), "tau": round(rng.uniform(0.05, 0.2), 3),
              "steps": rng.randint(1, 2), "inner": rng.randint(1, 3), "tol": 1e-11, "precision": "mixed"}
        return c
    n, r, low, shifts = rng.choice(HEATBATH if kind == "heatbath" else FORCE)
    precision = "fp64" if kind == "heatbath" else rng.choice(["mixed", "mixed", "fp64"])
    # columns x sites, so that an FP64 solve stays below the largest case
    most = 131072 * 8 if precision == "mixed" else 20000 * 4
    c |= _extents(rng, 256, max(1024, min(131072, most // n)))
    c |= {"n": n, "r": r, "low": low, "shifts": shifts, "mass": _mass(rng, low)}
    c["tol"] = 1e-14 if kind == "heatbath" else 1e-11 if precision == "mixed" else 1e-12
    if kind != "heatbath":
        c["precision"] = precision
    return c


# ---------------------------------------------------------------- inputs
def _dims(c):
    return c["lx"], c["ly"], c["lz"], c["lt"]


def _generator(seed, salt):
    return torch.Generator(device=DEV).manual_seed(int(seed) * 64 + salt)


def _normal(shape, seed, salt):
    return torch.randn(shape, dtype=torch.float64, device=DEV, generator=_generator(seed, salt))


def _gell_mann():
    lam = np.zeros((8, 3, 3), dtype=np.complex128)
    lam[0, 0, 1] = lam[0, 1, 0] = 1
    lam[1, 0, 1], lam[1, 1, 0] = -1j, 1j
    lam[2, 0, 0], lam[2, 1, 1] = 1, -1
    lam[3, 0, 2] = lam[3, 2, 0] = 1
    lam[4, 0, 2], lam[4, 2, 0] = -1j, 1j
    lam[5, 1, 2] = lam[5, 2, 1] = 1
    lam[6, 1, 2], lam[6, 2, 1] = -1j, 1j
    lam[7] = np.diag([1, 1, -2]) / math.sqrt(3)
    return torch.from_numpy(lam).to(DEV)


def _mm(a, b):
    """Product of 3 x 3 matrices held as (..., 3, 3)."""
    return sum(a[..., :, k:k + 1] * b[..., k:k + 1, :] for k in range(3))


def _exp(Y):
    """exp of 3 x 3 matrices in 64 bits: Taylor polynomial of Y / 64, squared six times."""
    Y = Y / 64
    eye = torch.eye(3, dtype=Y.dtype, device=Y.device).expand_as(Y)
    E = eye
    for k in range(14, 0, -1):
        E = eye + _mm(Y, E) / k
    for _ in range(6):
        E = _mm(E, E)
    return E


def _links(dims, eps, seed, salt=0):
    """exp(i eps H), H = sum_a h^a lambda^a / 2, h^a ~ N(0, 1): (Lt, Lz, Ly, Lx, 4, 3, 3)."""
    lx, ly, lz, lt = dims
    h = _normal((lt, lz, ly, lx, 4, 8), seed, salt).to(torch.complex128)
    return _exp((0.5j * eps) * (h @ _gell_mann().reshape(8, 9)).reshape(lt, lz, ly, lx, 4, 3, 3)).contiguous()


def _block(dims, n, seed, salt=1):
    """n complex Gaussian fields on one parity, density exp(-|phi|^2)."""
    vh = dims[0] * dims[1] * dims[2] * dims[3] // 2
    return torch.view_as_complex(_normal((vh, 3, n, 2), seed, salt) * math.sqrt(0.5)).contiguous()


def _members(c):
    """(dims, n, exponent) of a batch: extents first, first + 4, ...; n = 2, 4, 8 as in the batched workload."""
    return [((c["first"] + 4 * i,) * 4, 2 << i, -1.0 / (8 << i)) for i in range(c["members"])]


_last = [None]


def _one_lattice(key):
    """A program works on one lattice at a time: the contexts of the one before are given back."""
    if _last[0] != key:
        rhmc.clear_contexts()
        _last[0] = key


def _momenta(dims, seed, salt=2):
    lx, ly, lz, lt = dims
    return _normal((lt, lz, ly, lx, 4, 8), seed, salt)


def _trajectory_rationals(n):
    return rational_approx(1.0 / (8 * n), 2e-3, 64.0, 12), rational_approx(-1.0 / (4 * n), 2e-3, 64.0, 12)


def prepare(case, seed):
    c = dict(case)
    kind = c["kind"]
    s = {"case": c}
    if kind == "batch":
        _one_lattice(None)
        s["items"] = []
        for i, (dims, n, r) in enumerate(_members(c)):
            ctx = RhmcContext(dims, c["mass"])
            ctx.set_gauge(_links(dims, c["eps"], seed, 10 + i))
            s["items"].append((ctx, _block(dims, n, seed, 20 + i), rational_approx(r, c["low"], 64.0, c["shifts"]).beta))
        return s
    dims = _dims(c)
    U = _links(dims, c.get("eps", 0.5), seed)
    if kind == "operator":
        _one_lattice(None)
        s["ctx"] = RhmcContext(dims, c["mass"])
        s["ctx"].set_gauge(U)
        s["X"] = _block(dims, c["n"], seed)
        return s
    s["U"] = U
    if kind in ("md", "trajectory"):
        _one_lattice(None)
        s["ctx"] = RhmcContext(dims, c["mass"])
        p = _momenta(dims, seed)
        s["par"] = hmc.MdParams(beta=BETA, tau=c["tau"], n_steps=c["steps"], n_gauge=c["inner"], tol_md=c["tol"],
                                precision=c["precision"])
        if kind == "md":
            s["P"] = hmc.momenta(s["ctx"], p)
        else:
            s["p"], s["eta"] = p, _block(dims, c["n"], seed)
            s["hb"], s["ra"] = _trajectory_rationals(c["n"])
        return s
    _one_lattice((dims, c["mass"]))
    s["ra"] = rational_approx(c["r"], c["low"], 64.0, c["shifts"])
    s["Phi"] = _block(dims, c["n"], seed)
    return s


def run(s):
    c = s["case"]
    kind = c["kind"]
    if kind == "operator":
        return s["ctx"].apply_mdagm_mrhs(s["X"], 0.0, c["precision"])
    if kind == "batch":
        return [X for X, _ in block_multishift_cg_batch(s["items"], c["tol"], precision=c["precision"])]
    if kind == "md":
        U, P = s["U"].clone(), s["P"].clone()
        hmc.md_evolve(s["ctx"], U, P, None, None, s["par"])
        return {"U": U, "P": P}
    if kind == "trajectory":
        U = s["U"].clone()
        t = hmc.trajectory(s["ctx"], U, s["p"], s["eta"], s["hb"], s["ra"], s["ra"], s["par"], tol_action=1e-13,
                           u=0.0, want_phi=True)
        return {"U": U, "Phi": t["Phi"], "H_old": t["H_old"], "H_new": t["H_new"], "accepted": t["accepted"]}
    ra = s["ra"]
    if kind == "solve":
        return rhmc.block_multishift_cg(s["U"], s["Phi"], ra.beta, c["tol"], c["mass"], precision=c["precision"])[0]
    if kind == "force":
        G, S, _ = rhmc.force(s["U"], s["Phi"], ra, c["tol"], c["mass"], precision=c["precision"])
        return {"G": G, "S": S}
    if kind == "heatbath":
        ctx = rhmc.context_for(s["U"], c["mass"])
        return ctx.rational_solve(s["Phi"], ra.alpha0, ra.alpha, ra.beta, c["tol"])[0]
    U, Phi = s["U"].clone().requires_grad_(), s["Phi"].clone().requires_grad_()
    S = rhmc.PseudofermionAction.apply(U, Phi, ra, c["mass"], tol=c["tol"], precision=c["precision"])
    S.backward()
    return {"S": S.detach(), "U": U.grad, "Phi": Phi.grad}


# ---------------------------------------------------------------- what a pass cannot do without
def _solve_work(dims, n, mass, shifts, tol):
    """Operator flops of the iterations that a Krylov space of n columns needs: CG's bound, a half of it taken."""
    v = dims[0] * dims[1] * dims[2] * dims[3]
    its = 0.25 * math.sqrt(64.0 / (4 * mass * mass + 1e-4)) * math.log(2.0 / tol)
    return 16.0 * (v * 36 + v // 2 * 3 * n), its * (v // 2) * n * 2 * 576.0, v // 2 * 3 * n * 16.0


def work(case):
    c = dict(case)
    kind = c["kind"]
    if kind == "batch":
        b = f = 0.0
        for dims, n, _ in _members(c):
            x, y, field = _solve_work(dims, n, c["mass"], c["shifts"], c["tol"])
            b, f = b + x + c["shifts"] * field, f + y
        return {"bytes": b, "flops": f}
    dims = _dims(c)
    v = dims[0] * dims[1] * dims[2] * dims[3]
    links = v * 36 * 16.0
    if kind == "operator":
        return {"bytes": links + 2 * v // 2 * 3 * c["n"] * 16.0, "flops": v // 2 * c["n"] * 2 * 576.0}
    if kind == "md":  # per link: a kick of 9 matrix products, an update of 2 and the exponential's scalars
        kicks = 2 * c["steps"] * (2 * c["inner"] + 1)
        return {"bytes": 4 * links, "flops": v * 4 * 216.0 * kicks * 11}
    if kind == "trajectory":
        b, f, field = _solve_work(dims, c["n"], c["mass"], 12, c["tol"])
        kicks = 2 * c["steps"] * (2 * c["inner"] + 1)
        return {"bytes": b + links + field, "flops": f * (2 * c["steps"] + 1 + 3 * 1.3) + v * 4 * 216.0 * kicks * 11}
    b, f, field = _solve_work(dims, c["n"], c["mass"], c["shifts"], c["tol"])
    outer = v * 4 * 9 * c["shifts"] * c["n"] * 8.0
    return {"solve": {"bytes": b + c["shifts"] * field, "flops": f}, "heatbath": {"bytes": b + field, "flops": f},
            "force": {"bytes": b + links, "flops": f + outer},
            "action": {"bytes": b + links + field, "flops": f + outer}}[kind]


# ---------------------------------------------------------------- the same in plain torch, 64 bits
class _Lattice:
    def __init__(self, dims, U, mass):
        lx, ly, lz, lt = self.dims = dims
        self.mass, V = mass, lx * ly * lz * lt
        x = torch.arange(lx, device=DEV).view(1, 1, 1, lx)
        y = torch.arange(ly, device=DEV).view(1, 1, ly, 1)
        z = torch.arange(lz, device=DEV).view(1, lz, 1, 1)
        t = torch.arange(lt, device=DEV).view(lt, 1, 1, 1)
        lex = (x + lx * (y + ly * (z + lz * t)))
        odd = ((x + y + z + t) % 2).expand(lt, lz, ly, lx)
        zero = torch.zeros_like(lex)
        eta = [zero, zero + x, zero + x + y, zero + x + y + z]
        sign = [1.0 - 2.0 * (e % 2).double() for e in eta]
        sign[3] = torch.where(t == lt - 1, -sign[3], sign[3])  # antiperiodic in time
        self.sign, self.odd = torch.stack(sign, -1), odd
        self.sites = [torch.nonzero(odd.reshape(-1) == p).reshape(-1) for p in (0, 1)]
        self.up = [torch.roll(lex, -1, 3 - mu).reshape(-1) for mu in range(4)]
        W = (U * self.sign[..., None, None]).reshape(V, 4, 3, 3)
        self.rank = [s // 2 for s in self.sites]
        self.hops = []  # for each output parity: (matrix, input rank) of the eight neighbours
        down = [torch.roll(lex, 1, 3 - mu).reshape(-1) for mu in range(4)]
        for p in (0, 1):
            at = self.sites[p]
            h = [(W[at, mu], self.up[mu][at] // 2) for mu in range(4)]
            h += [(-W[down[mu][at], mu].conj().transpose(-1, -2), down[mu][at] // 2) for mu in range(4)]
            self.hops.append([(m.contiguous(), i) for m, i in h])

    def hop(self, X, p):
        out = 0
        for m, i in self.hops[p]:
            v = X[i]
            out = out + sum(m[:, :, k, None] * v[:, k, None, :] for k in range(3))
        return out

    def apply(self, X, sigma=0.0):
        return (4 * self.mass ** 2 + sigma) * X - self.hop(self.hop(X, 1), 0)

    def solve(self, B, shifts, weights=None):
        """Multishift CG, every column with scalars of its own.  The solutions, or their weighted sum."""
        order = sorted(range(len(shifts)), key=lambda q: shifts[q])
        sh = torch.tensor([shifts[q] for q in order], dtype=torch.float64, device=DEV)
        ns, n, tol = len(shifts), B.shape[-1], 3e-15
        col = lambda a: a.view(ns, 1, 1, n)  # noqa: E731
        dot = lambda a, b: torch.einsum("vcn,vcn->n", a.conj(), b).real  # noqa: E731
        X = torch.zeros((ns,) + B.shape, dtype=B.dtype, device=DEV)
        P, r = B.repeat(ns, 1, 1, 1), B.clone()
        rr = dot(r, r)
        bb = rr.clone()
        zeta = torch.ones(ns, n, dtype=torch.float64, device=DEV)
        before, a0, b0 = zeta.clone(), torch.ones_like(rr), torch.zeros_like(rr)
        ds = (sh - sh[0])[:, None]
        for k in range(6000):
            Ap = self.apply(P[0], float(sh[0]))
            a = rr / dot(P[0], Ap)
            after = zeta * before * a0 / (a0 * before * (1 + ds * a) + a * b0 * (before - zeta))
            after = torch.where(after.abs() < 1e-200, torch.zeros_like(after), after)
            ratio = torch.where(zeta == 0, torch.zeros_like(zeta), after / torch.where(zeta == 0, 1.0, zeta))
            X += col(a * ratio) * P
            r -= a * Ap
            new = dot(r, r)
            b = new / rr
            P.mul_(col(b * ratio * ratio)).add_(col(after) * r)
            before, zeta, a0, b0, rr = torch.where(zeta == 0, 1.0, zeta), after, a, b, new
            if k % 20 == 19 and float((new / bb).max()) < tol * tol:
                break
        if weights is not None:
            return sum(weights[order[q]] * X[q] for q in range(ns))
        out = torch.empty_like(X)
        for q in range(ns):
            out[order[q]] = X[q]
        return out

    def force(self, X, alpha):
        """G_mu(x) = 2 eps eta b sum_s alpha_s W_s(x) W_s(x + mu)^dagger, W = X on even, D_oe X on odd sites."""
        V = 2 * X.shape[1]
        G = torch.zeros((V, 4, 3, 3), dtype=X.dtype, device=DEV)
        for q, a in enumerate(alpha):
            W = torch.empty((V,) + X.shape[2:], dtype=X.dtype, device=DEV)
            W[self.sites[0]], W[self.sites[1]] = X[q], self.hop(X[q], 1)
            for mu in range(4):
                w = W[self.up[mu]].conj()
                G[:, mu] += a * torch.stack([(W[:, i, None, :] * w).sum(-1) for i in range(3)], 1)
        parity = (1.0 - 2.0 * self.odd.reshape(-1).double())
        return 2.0 * (parity[:, None] * self.sign.reshape(V, 4))[..., None, None] * G


def _dagger(m):
    return m.conj().transpose(-1, -2)


def _traceless(m):
    m = (m - _dagger(m)) / 2
    tr = m.diagonal(dim1=-2, dim2=-1).sum(-1) / 3
    return m - tr[..., None, None] * torch.eye(3, dtype=m.dtype, device=m.device)


def _shift(U, mu, d):
    return torch.roll(U, -d, 3 - mu)


def _gauge_kick(U, P, eps):
    """P += eps TA(U G^dagger) / 2 with the Wilson action's derivative G = -(beta / 3) V^dagger, V the staples."""
    for mu in range(4):
        V = 0
        for nu in range(4):
            if nu == mu:
                continue
            un, um = U[..., nu, :, :], U[..., mu, :, :]
            V = V + _mm(_mm(_shift(un, mu, 1), _dagger(_shift(um, nu, 1))), _dagger(un))
            d = _shift(_shift(un, mu, 1), nu, -1)
            V = V + _mm(_dagger(_mm(_shift(um, nu, -1), d)), _shift(un, nu, -1))
        P[..., mu, :, :] -= (eps * BETA / 6) * _traceless(_mm(U[..., mu, :, :], V))


def _gauge_energy(U):
    S = 0.0
    for mu in range(4):
        for nu in range(mu + 1, 4):
            um, un = U[..., mu, :, :], U[..., nu, :, :]
            a, b = _mm(um, _shift(un, mu, 1)), _mm(un, _shift(um, nu, 1))
            S += BETA * (1.0 - (a * b.conj()).sum((-1, -2)).real / 3).sum()
    return float(S)


def _evolve(c, U, P, kick):
    """Two-level OMF2: `kick` outside, the gauge force in `inner` steps of each half step."""
    lam, e = 1.0 / 6, c["tau"] / c["steps"]

    def drift(U, h):
        h = h / c["inner"]
        for _ in range(c["inner"]):
            _gauge_kick(U, P, lam * h)
            U = _mm(_exp(0.5 * h * P), U)
            _gauge_kick(U, P, (1 - 2 * lam) * h)
            U = _mm(_exp(0.5 * h * P), U)
            _gauge_kick(U, P, lam * h)
        return U

    for _ in range(c["steps"]):
        kick(U, lam * e)
        U = drift(U, 0.5 * e)
        kick(U, (1 - 2 * lam) * e)
        U = drift(U, 0.5 * e)
        kick(U, lam * e)
    return U


def _algebra(p):
    return ((0.5j * p.to(torch.complex128)) @ _gell_mann().reshape(8, 9)).reshape(p.shape[:-1] + (3, 3))


def exact(case, seed):
    c = dict(case)
    kind = c["kind"]
    if kind == "batch":
        if c["first"] + 4 * (c["members"] - 1) > 18:
            return None
        out = []
        for i, (dims, n, r) in enumerate(_members(c)):
            L = _Lattice(dims, _links(dims, c["eps"], seed, 10 + i), c["mass"])
            out.append(L.solve(_block(dims, n, seed, 20 + i), rational_approx(r, c["low"], 64.0, c["shifts"]).beta))
        return out
    dims = _dims(c)
    v = dims[0] * dims[1] * dims[2] * dims[3]
    U = _links(dims, c.get("eps", 0.5), seed)
    if kind == "operator":
        return _Lattice(dims, U, c["mass"]).apply(_block(dims, c["n"], seed))
    if kind == "md":
        P = _algebra(_momenta(dims, seed))
        return {"U": _evolve(c, U, P, lambda u, e: None), "P": P}
    if kind == "trajectory":
        hb, ra = _trajectory_rationals(c["n"])
        P, eta = _algebra(_momenta(dims, seed)), _block(dims, c["n"], seed)
        start = _Lattice(dims, U, c["mass"])
        Phi = hb.alpha0 * eta + start.solve(eta, hb.beta, hb.alpha)

        def energy(L, U):
            R = ra.alpha0 * Phi + L.solve(Phi, ra.beta, ra.alpha)
            return float((Phi.conj() * R).sum().real) + _gauge_energy(U) - float((P * P.transpose(-1, -2)).sum().real)

        def kick(u, e):
            L = _Lattice(dims, u, c["mass"])
            G = L.force(L.solve(Phi, ra.beta), ra.alpha).reshape(u.shape)
            P.add_(0.5 * e * _traceless(_mm(u, _dagger(G))))

        old = energy(start, U)
        U = _evolve(c, U, P, kick)
        return {"U": U, "Phi": Phi, "H_old": old, "H_new": energy(_Lattice(dims, U, c["mass"]), U), "accepted": None}
    if v * c["n"] * c["shifts"] > 131072 * 8 * 16:  # longer than about 20 seconds
        return None
    L, Phi, ra = _Lattice(dims, U, c["mass"]), _block(dims, c["n"], seed), rational_approx(c["r"], c["low"], 64.0, c["shifts"])
    if kind == "heatbath":
        return ra.alpha0 * Phi + L.solve(Phi, ra.beta, ra.alpha)
    X = L.solve(Phi, ra.beta)
    if kind == "solve":
        return X
    R = ra.alpha0 * Phi + sum(a * X[q] for q, a in enumerate(ra.alpha))
    S, G = float((Phi.conj() * R).sum().real), L.force(X, ra.alpha)
    if kind == "force":
        return {"G": G, "S": S}
    S = torch.tensor(S, dtype=torch.float64)
    return {"S": S, "U": G.reshape(U.shape), "Phi": 2 * R}
