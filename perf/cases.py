"""Performance cases: the calls a user of this framework makes, through its public entry points.

Kinds of calls
  aimd      one AIMD step there and one back: the nuclei move by a velocity-Verlet step of
            0.5 fs, rihf_update_geometry + rihf_scf from the previous orbitals + rihf_gradient,
            then the same back to the first geometry (so every pass does the same work)
  point     a cold single point: new geometry, SCF from a cold guess, density and orbital
            energies read back, analytic gradient
  batch     one AIMD step there and one back of a batch of independent clusters
  integrals new geometry, then S, h, (P|Q) and (mu nu|P) read back: what a program that
            brings its own method takes from this library

Sizes, basis sets and thresholds are those of the workloads module, the tests and the
benchmark.  Contexts, like a user's program, are kept between calls; nothing else is.
"""

from __future__ import annotations

import math

import numpy as np
import torch

from paper_2407_19614_gb300 import rihf as R
from paper_2407_19614_gb300 import workloads as W

DT = 0.5 * W.FS_TO_AU
CONV = dict(conv_e=1e-8, conv_diis=1e-7, max_iter=100)          # AIMD thresholds of the benchmark
CONV_LARGE = dict(conv_e=1e-8, conv_diis=1e-6, max_iter=100, lindep_tau=1e-6)   # larger basis, 5 waters or more
CONV_LARGE_FEW = dict(conv_e=1e-10, conv_diis=1e-8, max_iter=100)   # larger basis, monomer to trimer
TIGHT = dict(conv_e=1e-10, conv_diis=1e-9, max_iter=100)         # a careful single point
EXACT_MOST = 200   # largest N that exact() takes


def listed():
    return [
        # smallest call: one water from scratch in FP64; launches and latency count
        dict(name="point_water1_fp64", kind="point", n=1, basis="small", precision="fp64", pure=True, contracted=False, guess=0),
        # Cartesian functions and contracted shells, the other options of a basis set
        dict(name="point_water2_cartesian", kind="point", n=2, basis="small", precision="fp64", pure=False, contracted=True, guess=5),
        # integrals alone, f and g functions
        dict(name="integrals_water1_large", kind="integrals", n=1, basis="large", precision="fp64", pure=True, contracted=False, guess=0),
        # AIMD of a small cluster, where each step is short
        dict(name="aimd_water3_mixed", kind="aimd", n=3, basis="small", precision="mixed", pure=True, contracted=False, guess=2),
        # the benchmark's AIMD step, on the mixed and on the FP64 path
        dict(name="aimd_water8_mixed", kind="aimd", n=8, basis="small", precision="mixed", pure=True, contracted=False, guess=2),
        dict(name="aimd_water8_fp64", kind="aimd", n=8, basis="small", precision="fp64", pure=True, contracted=False, guess=2),
        # a cluster above the one-CTA eigensolver's order (N = 384)
        dict(name="aimd_water16_mixed", kind="aimd", n=16, basis="small", precision="mixed", pure=True, contracted=False, guess=2),
        # the larger basis (f primary, g auxiliary): a small cluster, and the largest call
        dict(name="point_water3_large_mixed", kind="point", n=3, basis="large", precision="mixed", pure=True, contracted=False, guess=5),
        dict(name="point_water10_large_mixed", kind="point", n=10, basis="large", precision="mixed", pure=True, contracted=False, guess=5),
        # many small clusters at once, ragged sizes
        dict(name="batch_16x3to6_mixed", kind="batch", n=6, lo=3, count=16, basis="small", precision="mixed", pure=True, contracted=False, guess=2),
    ]


def draw(rng):
    kind = rng.choice(["aimd", "aimd", "aimd", "point", "point", "integrals", "batch"])
    case = dict(kind=kind, basis="small", precision="mixed", pure=True, contracted=False, guess=2)
    if kind == "aimd":
        case["n"] = int(round(math.exp(rng.uniform(0.0, math.log(16.4)))))
        case["precision"] = "mixed" if case["n"] > 8 else rng.choice(["mixed", "mixed", "fp64"])
    elif kind == "point":
        case["basis"] = rng.choice(["small", "large"])
        # the larger basis: its overlap has eigenvalues around every threshold at 4 waters, where SCFs stall
        case["n"] = rng.choice([1, 2, 3, 3, 5, 6, 7, 8]) if case["basis"] == "large" else int(round(math.exp(rng.uniform(0.0, math.log(12.4)))))
        case["guess"] = 5
        case["precision"] = "mixed" if case["n"] > 5 else rng.choice(["mixed", "fp64"])
        if case["basis"] == "small" and case["n"] <= 4:
            case["pure"], case["contracted"] = rng.choice([(True, False), (True, True), (False, True), (False, False)])
    elif kind == "integrals":
        case["basis"] = rng.choice(["small", "large"])
        case["n"] = rng.randint(1, 2 if case["basis"] == "large" else 3)
        case["precision"], case["guess"] = "fp64", 0
        case["pure"] = rng.choice([True, True, False])
        case["contracted"] = case["basis"] == "small" and rng.choice([True, False])
    else:
        case["lo"] = rng.randint(1, 4)
        case["n"] = case["lo"] + rng.randint(0, 4)
        case["count"] = rng.randint(4, 20)
    case["tag"] = rng.randrange(1 << 30)   # this case's own cluster geometries
    return case


# ------------------------------------------------------------------ inputs

def _contract(shells, ratios, coefs):
    return [W.Shell(s.atom, s.l, [s.exps[0] * r for r in ratios], list(coefs)) for s in shells]


def _molecule(case, n, seed):
    mol = W.water_n(n, seed, case["basis"])
    if case["contracted"]:   # three primitives per primary shell, two per auxiliary shell
        mol.primary = _contract(mol.primary, (0.7, 1.0, 2.1), (0.3, 0.6, 0.25))
        mol.aux = _contract(mol.aux, (1.0, 1.6), (0.7, 0.4))
    return mol


def _options(case):
    if case["basis"] == "large":
        kw = dict(CONV_LARGE if case["n"] >= 5 else CONV_LARGE_FEW)
    else:
        kw = dict(CONV if case["kind"] in ("aimd", "batch") or case["precision"] == "mixed" else TIGHT)
    if case["precision"] == "mixed":
        kw["precision"] = R.PRECISION_MIXED
    kw["pure"] = 1 if case["pure"] else 0
    return kw


def _molecules(case, seed):
    rng = np.random.Generator(np.random.PCG64([int(seed), int(case.get("tag", 0))]))
    seeds = rng.integers(0, 1 << 31, size=64)
    if case["kind"] != "batch":
        return [_molecule(case, case["n"], int(seeds[0]))]
    sizes = [case["lo"] + i % (case["n"] - case["lo"] + 1) for i in range(case["count"])]
    return [_molecule(case, n, int(seeds[i])) for i, n in enumerate(sizes)]


def _moved(mol, grad, seed):
    """One velocity-Verlet step of 0.5 fs from 300 K velocities."""
    m = W.masses_au(mol.Z)[:, None]
    return mol.xyz + W.maxwell_boltzmann(mol.Z, 300.0, seed) * DT - 0.5 * grad / m * DT * DT


def prepare(case, seed):
    mols = _molecules(case, seed)
    ctx = [R.Context(m, **_options(case)) for m in mols]
    state = dict(kind=case["kind"], guess=case["guess"], ctx=ctx, x0=[m.xyz for m in mols])
    if case["kind"] in ("aimd", "batch"):
        state["x1"] = []
        for k, (m, c) in enumerate(zip(mols, ctx)):
            c.scf(guess=5, outputs=False)
            state["x1"].append(_moved(m, c.gradient(), int(seed) % 100003 + k))
    return state


# ------------------------------------------------------------------ passes

def run(state):
    kind, ctx = state["kind"], state["ctx"]
    if kind == "batch":
        out = []
        for xyz in (state["x1"], state["x0"]):
            energies, grads, _ = R.batch_step(ctx, xyz, guess=state["guess"])
            out.append(dict(energy=energies, grad=np.concatenate(grads)))
        return out
    c = ctx[0]
    if kind == "aimd":
        out = []
        for x in (state["x1"][0], state["x0"][0]):
            c.update_geometry(x)
            e = c.scf(guess=state["guess"], outputs=False)["energy"]
            out.append(dict(energy=np.array([e]), grad=c.gradient()))
        return out
    c.update_geometry(state["x0"][0])
    if kind == "integrals":
        return dict(S=c.matrix("S"), H=c.matrix("H"), A=c.matrix("A"), T3=c.matrix("T3"))
    r = c.scf(guess=state["guess"])
    return dict(energy=np.array([r["energy"]]), D=r["D"], eps=r["eps"], grad=c.gradient())


# ------------------------------------------------------------------ work and tolerance

def _sizes(case, n):
    small = case["basis"] == "small"
    if case["pure"]:
        return (24, 106, 5) if small else (58, 170, 5)
    return (25, 120, 5) if small else (65, 205, 5)


def work(case):
    """What one pass cannot do without: the fitted tensor is written once and read by every
    SCF iteration's J (and K), the fit and the RI-K products are made, per geometry."""
    ns = [case["n"]] if case["kind"] != "batch" else [case["lo"] + i % (case["n"] - case["lo"] + 1) for i in range(case["count"])]
    bytes_, flops = 0.0, 0.0
    for n in ns:
        N, NA, no = (n * v for v in _sizes(case, n))
        tri = N * (N + 1) / 2
        t3 = 8.0 * NA * tri
        if case["kind"] == "integrals":
            bytes_ += t3 + 8.0 * (NA * NA + 2 * N * N)
            flops += 600.0 * NA * tri / 4 + NA * NA * tri
            continue
        iters = 12
        steps = 2 if case["kind"] in ("aimd", "batch") else 1
        bytes_ += steps * (3 * t3 + iters * t3)
        flops += steps * (NA * NA * tri * 1.0 + (iters + 1) * 3.0 * NA * N * N * no + 600.0 * NA * tri / 4)
    return {"bytes": bytes_, "flops": flops}


def tolerance(case):
    if case["kind"] == "integrals":
        return {"rel": 1e-12, "max": 1e-10}   # FP64 recursions in another order, cancelling in small elements
    # SCF results: the last iterate is anywhere below the convergence thresholds, and these
    # nearly dependent sets turn rounding of the orbitals into changes of D and the forces
    if case["basis"] == "large":
        return {"rel": 5e-4, "max": 1e-2}
    if case["kind"] == "point" and case["precision"] == "fp64":
        return {"rel": 5e-6, "max": 2e-4}
    return {"rel": 2e-5, "max": 1e-3}


# ------------------------------------------------------------------ the same in plain torch, 64 bits

class _Boys(torch.autograd.Function):
    """F_0..F_n(T): the ascending series of F_n and downward recursion below T = 30, erf and
    upward recursion above (dF_m/dT = -F_{m+1})."""

    @staticmethod
    def forward(ctx, T, n):
        top = n + 1
        Ts = T.clamp(max=30.0)
        term = torch.full_like(Ts, 1.0 / (2 * top + 1))
        s = term.clone()
        for k in range(1, 160):
            term = term * (2.0 * Ts) / (2 * top + 2 * k + 1)
            s += term
        ex = torch.exp(-Ts)
        lo = [None] * (top + 1)
        lo[top] = ex * s
        for m in range(top - 1, -1, -1):
            lo[m] = (2.0 * Ts * lo[m + 1] + ex) / (2 * m + 1)
        Tl = T.clamp(min=30.0)
        ex = torch.exp(-Tl)
        hi = [0.5 * torch.sqrt(math.pi / Tl) * torch.erf(torch.sqrt(Tl))]
        for m in range(top):
            hi.append(((2 * m + 1) * hi[m] - ex) / (2.0 * Tl))
        F = torch.stack([torch.where(T < 30.0, a, b) for a, b in zip(lo, hi)])
        ctx.save_for_backward(F)
        return F[:-1]

    @staticmethod
    def backward(ctx, g):
        (F,) = ctx.saved_tensors
        return -(g * F[1:]).sum(0), None


def _carts(l):
    return [(x, y, l - x - y) for x in range(l, -1, -1) for y in range(l - x, -1, -1)]


def _herm(L):
    return [(t, u, v) for t in range(L + 1) for u in range(L + 1 - t) for v in range(L + 1 - t - u)]


def _harmonics(l):
    """Real solid harmonics S_lm, m = -l..l, as {(i, j, k): coefficient} (standard recursion in l)."""
    def mul(p, d, f=1.0):
        return {(a + d[0], b + d[1], c + d[2]): f * v for (a, b, c), v in p.items()}

    def add(*ps):
        out = {}
        for p in ps:
            for k, v in p.items():
                out[k] = out.get(k, 0.0) + v
        return out

    S = [{0: {(0, 0, 0): 1.0}}]
    for j in range(l):
        top, bot = S[j][j], S[j][-j]
        f = math.sqrt((2.0 if j == 0 else 1.0) * (2 * j + 1) / (2 * j + 2))
        new = {j + 1: mul(top, (1, 0, 0), f), -j - 1: mul(top, (0, 1, 0), f)}
        if j:
            new[j + 1] = add(new[j + 1], mul(bot, (0, 1, 0), -f))
            new[-j - 1] = add(new[-j - 1], mul(bot, (1, 0, 0), f))
        for m in range(-j, j + 1):
            p = mul(S[j][m], (0, 0, 1), 2 * j + 1)
            if abs(m) < j:
                q, g = S[j - 1][m], -math.sqrt((j + m) * (j - m))
                p = add(p, mul(q, (2, 0, 0), g), mul(q, (0, 2, 0), g), mul(q, (0, 0, 2), g))
            d = math.sqrt((j + m + 1) * (j - m + 1))
            new[m] = {k: v / d for k, v in p.items()}
        S.append(new)
    return [S[l][m] for m in range(-l, l + 1)]


class _Basis:
    """Primitive Cartesian functions grouped by l, and U: normalised contracted functions x primitives."""

    def __init__(self, shells, pure, dev):
        lmax = max(s.l for s in shells)
        self.groups, at = [], 0
        for l in range(lmax + 1):
            pr = [(i, s.atom, s.exps[k], s.coefs[k]) for i, s in enumerate(shells) if s.l == l for k in range(len(s.exps))]
            if not pr:
                continue
            n = len(pr) * len(_carts(l))
            self.groups.append(dict(l=l, sl=slice(at, at + n), shell=[p[0] for p in pr], coef=[p[3] for p in pr],
                                    atom=torch.tensor([p[1] for p in pr], device=dev),
                                    exp=torch.tensor([p[2] for p in pr], dtype=torch.float64, device=dev)))
            at += n
        self.n = at
        first, nf = [], 0
        for s in shells:
            first.append(nf)
            nf += 2 * s.l + 1 if pure else len(_carts(s.l))
        U = np.zeros((nf, at))
        for g in self.groups:
            l, cs = g["l"], _carts(g["l"])
            rows = _harmonics(l) if pure else [{c: 1.0} for c in cs]
            for q, (sh, co, a) in enumerate(zip(g["shell"], g["coef"], g["exp"].tolist())):
                for r, poly in enumerate(rows):
                    for c, v in poly.items():
                        U[first[sh] + r, g["sl"].start + q * len(cs) + cs.index(c)] += v * co * a ** (0.5 * l + 0.75) * 2.0 ** l
        self.U = torch.tensor(U, device=dev)


def _e_table(la, lb, PA, PB, inv2p, E0):
    """Hermite expansion coefficients E_t^{ij} of one dimension, t = 0..i+j."""
    E = {(0, 0): [E0]}

    def raise_(e, d):
        out = []
        for t in range(len(e) + 1):
            v = inv2p * e[t - 1] if t >= 1 else 0.0
            if t < len(e):
                v = v + d * e[t]
            if t + 1 < len(e):
                v = v + (t + 1) * e[t + 1]
            out.append(v if torch.is_tensor(v) else torch.zeros_like(E0))
        return out

    for i in range(la + 1):
        if i:
            E[i, 0] = raise_(E[i - 1, 0], PA)
        for j in range(1, lb + 1):
            E[i, j] = raise_(E[i, j - 1], PB)
    return E


def _pair(ga, gb, x):
    """All primitive pairs of two groups: p, P, and the E matrix (pair, cartesian a b, hermite)."""
    a = ga["exp"].repeat_interleave(len(gb["exp"]))
    b = gb["exp"].repeat(len(ga["exp"]))
    A, B = x[ga["atom"]].repeat_interleave(len(gb["exp"]), 0), x[gb["atom"]].repeat(len(ga["exp"]), 1)
    p = a + b
    P = (a[:, None] * A + b[:, None] * B) / p[:, None]
    la, lb = ga["l"], gb["l"]
    tabs = [_e_table(la, lb, P[:, d] - A[:, d], P[:, d] - B[:, d], 0.5 / p, torch.exp(-a * b / p * (A[:, d] - B[:, d]) ** 2))
            for d in range(3)]
    hs = _herm(la + lb)
    zero = torch.zeros_like(p)
    rows = []
    for ca in _carts(la):
        for cb in _carts(lb):
            e = [tabs[d][ca[d], cb[d]] for d in range(3)]
            rows.append(torch.stack([e[0][h[0]] * e[1][h[1]] * e[2][h[2]] if all(h[d] < len(e[d]) for d in range(3)) else zero
                                     for h in hs], -1))
    return p, P, torch.stack(rows, 1), tabs, (a, b)


def _single(g, x):
    """One group as a pair with a unit s function."""
    q = g["exp"]
    zero = torch.zeros_like(q)
    tabs = _e_table(g["l"], 0, zero, zero, 0.5 / q, torch.ones_like(q))
    hs = _herm(g["l"])
    rows = [torch.stack([math.prod(tabs[c[d], 0][h[d]] for d in range(3)) if all(h[d] <= c[d] for d in range(3)) else zero
                         for h in hs], -1) for c in _carts(g["l"])]
    return q, x[g["atom"]], torch.stack(rows, 1)


def _coulomb(p, P, lp, q, Q, lq):
    """(pair, hermite of p, hermite of q) Hermite Coulomb integrals over all pairs of the two lists."""
    L = lp + lq
    X = P[:, None, :] - Q[None, :, :]
    rho = p[:, None] * q[None, :] / (p[:, None] + q[None, :]) if q is not None else p[:, None].expand(X.shape[:2])
    F = _Boys.apply(rho * (X * X).sum(-1), L)
    Rn = {(0, 0, 0): [(-2.0 * rho) ** n * F[n] for n in range(L + 1)]}
    for tot in range(1, L + 1):
        for h in _herm(L):
            if sum(h) != tot:
                continue
            d = next(k for k in range(3) if h[k])
            h1 = tuple(h[k] - (k == d) for k in range(3))
            h2 = tuple(h[k] - 2 * (k == d) for k in range(3))
            Rn[h] = [X[..., d] * Rn[h1][n + 1] + ((h[d] - 1) * Rn[h2][n + 1] if h[d] > 1 else 0.0) for n in range(L + 1 - tot)]
    return torch.stack([torch.stack([(-1.0) ** sum(k) * Rn[h[0] + k[0], h[1] + k[1], h[2] + k[2]][0] for k in _herm(lq)], -1)
                        for h in _herm(lp)], -2)


class _Exact:
    """Integrals of one molecule over primitives; weights: {name: matrix over primitives} to
    contract with instead (a scalar whose backward pass is the gradient)."""

    def __init__(self, mol, pure, dev):
        self.Z = torch.tensor(mol.Z, dtype=torch.float64, device=dev)
        self.p, self.a = _Basis(mol.primary, pure, dev), _Basis(mol.aux, pure, dev)
        self.dev = dev
        x = torch.tensor(mol.xyz, dtype=torch.float64, device=dev)
        with torch.no_grad():
            for b in (self.p, self.a):   # every contracted function normalised to one
                s = b.U @ self._overlap(b, x)[0] @ b.U.T
                b.U = b.U / torch.sqrt(torch.diagonal(s))[:, None]

    def _overlap(self, b, x, parts=False):
        S = torch.zeros((b.n, b.n), dtype=torch.float64, device=self.dev)
        T = torch.zeros_like(S)
        for ga in b.groups:
            for gb in b.groups:
                la, lb = ga["l"], gb["l"]
                up = dict(gb, l=lb + 2)
                p, _, _, tabs, (_, be) = _pair(ga, up, x) if parts else _pair(ga, gb, x)
                f = torch.sqrt(math.pi / p)
                s = lambda d, i, j: tabs[d][i, j][0] * f if j >= 0 else 0.0
                sb, tb = [], []
                for ca in _carts(la):
                    for cb in _carts(lb):
                        s0 = [s(d, ca[d], cb[d]) for d in range(3)]
                        sb.append(s0[0] * s0[1] * s0[2])
                        if parts:
                            k0 = [4 * be * be * s(d, ca[d], cb[d] + 2) - 2 * be * (2 * cb[d] + 1) * s0[d]
                                  + cb[d] * (cb[d] - 1) * s(d, ca[d], cb[d] - 2) for d in range(3)]
                            tb.append(-0.5 * (k0[0] * s0[1] * s0[2] + s0[0] * k0[1] * s0[2] + s0[0] * s0[1] * k0[2]))
                shape = (len(ga["exp"]), len(gb["exp"]), len(_carts(la)), len(_carts(lb)))
                n, m = shape[0] * shape[2], shape[1] * shape[3]
                S[ga["sl"], gb["sl"]] = torch.stack(sb, -1).reshape(shape).permute(0, 2, 1, 3).reshape(n, m)
                if parts:
                    T[ga["sl"], gb["sl"]] = torch.stack(tb, -1).reshape(shape).permute(0, 2, 1, 3).reshape(n, m)
        return S, T

    def _blocks(self, x):
        """Yields (kind, slices, block) of V, (P|Q) and (mu nu|P) over primitives."""
        for ia, ga in enumerate(self.p.groups):
            for gb in self.p.groups[: ia + 1]:
                p, P, E, _, _ = _pair(ga, gb, x)
                la, lb = ga["l"], gb["l"]
                sh = (len(ga["exp"]), len(gb["exp"]), len(_carts(la)), len(_carts(lb)))
                Rv = _coulomb(p, P, la + lb, None, x, 0)[..., 0]
                v = torch.einsum("kat,kct,c,k->ka", E, Rv, -self.Z, 2 * math.pi / p)
                yield "V", (ga["sl"], gb["sl"]), v.reshape(sh).permute(0, 2, 1, 3).reshape(sh[0] * sh[2], sh[1] * sh[3])
                for gc in self.a.groups:
                    q, Q, Ec = _single(gc, x)
                    f = 2 * math.pi ** 2.5 / (p[:, None] * q[None] * torch.sqrt(p[:, None] + q[None]))
                    r = _coulomb(p, P, la + lb, q, Q, gc["l"])
                    t = torch.einsum("kat,kcts->kcas", E, r * f[..., None, None])
                    t = torch.einsum("kcas,cds->cdka", t, Ec)
                    yield "T3", (gc["sl"], ga["sl"], gb["sl"]), t.reshape((-1,) + sh).permute(0, 1, 3, 2, 4).reshape(
                        -1, sh[0] * sh[2], sh[1] * sh[3])
        for ia, ga in enumerate(self.a.groups):
            p, P, E = _single(ga, x)
            for gc in self.a.groups[: ia + 1]:
                q, Q, Ec = _single(gc, x)
                f = 2 * math.pi ** 2.5 / (p[:, None] * q[None] * torch.sqrt(p[:, None] + q[None]))
                r = _coulomb(p, P, ga["l"], q, Q, gc["l"]) * f[..., None, None]
                b = torch.einsum("kat,kcts,cds->kacd", E, r, Ec)
                yield "A", (ga["sl"], gc["sl"]), b.reshape(b.shape[0] * b.shape[1], -1)

    def matrices(self, x):
        with torch.no_grad():
            Up, Ua = self.p.U, self.a.U
            S, T = self._overlap(self.p, x, True)
            V, A = torch.zeros_like(S), torch.zeros((self.a.n, self.a.n), dtype=torch.float64, device=self.dev)
            T3 = torch.zeros((self.a.n, self.p.n, self.p.n), dtype=torch.float64, device=self.dev)
            full = {"V": V, "A": A, "T3": T3}
            for k, sl, b in self._blocks(x):
                full[k][sl] = b
                full[k][sl[:-2] + (sl[-1], sl[-2])] = b.transpose(-1, -2)
            T3 = torch.einsum("pmn,an->pma", T3, Up)
            T3 = torch.einsum("pma,bm->pba", T3, Up)
            T3 = (Ua @ T3.reshape(T3.shape[0], -1)).reshape(-1, Up.shape[0], Up.shape[0])
            return Up @ S @ Up.T, Up @ (T + V) @ Up.T, Ua @ A @ Ua.T, T3

    def gradient(self, x, D, Wm, Y, Zm):
        Up, Ua = self.p.U, self.a.U
        x = x.clone().requires_grad_(True)
        Dp, Wp = Up.T @ D @ Up, Up.T @ Wm @ Up
        w = {"V": Dp, "A": -0.5 * Ua.T @ Zm @ Ua}
        Yp = torch.einsum("pba,bm,an->pmn", Y, Up, Up)
        w["T3"] = (Ua.T @ Yp.reshape(Yp.shape[0], -1)).reshape(-1, self.p.n, self.p.n)
        S, T = self._overlap(self.p, x, True)
        r = torch.sqrt(((x[:, None] - x[None]) ** 2).sum(-1) + torch.eye(len(x), device=self.dev))
        zz = self.Z[:, None] * self.Z[None]
        nn = 0.5 * (zz / r * (1 - torch.eye(len(x), device=self.dev))).sum()
        ((Dp * T).sum() - (Wp * S).sum() + nn).backward()
        for k, sl, b in self._blocks(x):
            two = 1.0 if sl[-1] == sl[-2] else 2.0
            (two * (w[k][sl] * b).sum()).backward(retain_graph=True)   # the pair tables are shared
        return x.grad


def _solve(ex, x, nocc, lindep, C0=None):
    """RI-HF to convergence: (energy, D, eps, gradient, occupied orbitals)."""
    S, h, A, T3 = ex.matrices(x)
    N = S.shape[0]
    # by substitution on the host: GPU libraries invert diagonal blocks, which cond(A) = 1e9 does not forgive
    Lc = torch.linalg.cholesky(A.cpu())
    tri = lambda M, v, up: torch.linalg.solve_triangular(M, v.cpu().reshape(v.shape[0], -1), upper=up).reshape(v.shape).to(v.device)
    B = tri(Lc, T3, False)
    s, U = torch.linalg.eigh(S)
    X = U[:, s > lindep] / torch.sqrt(s[s > lindep])
    for _ in range(2):   # X^T S X = 1 to rounding, which eigenvectors of small overlap eigenvalues alone miss
        X = X @ (1.5 * torch.eye(X.shape[1], dtype=X.dtype, device=X.device) - 0.5 * X.T @ S @ X)
    if C0 is None:   # generalised Wolfsberg-Helmholz
        d = torch.diagonal(h)
        F = 0.875 * S * (d[:, None] + d[None])
        F[torch.arange(N), torch.arange(N)] = d
    else:
        M = torch.linalg.cholesky(C0.T @ S @ C0)
        Co = torch.linalg.solve_triangular(M, C0.T, upper=False).T
        F = None
    enuc = 0.0
    xs = x.cpu().numpy()
    Zs = ex.Z.cpu().numpy()
    for i in range(len(Zs)):
        for j in range(i):
            enuc += Zs[i] * Zs[j] / np.linalg.norm(xs[i] - xs[j])
    fs, es, best, stalled = [], [], 1e300, 0
    for it in range(150):
        if F is not None:
            eps, Cp = torch.linalg.eigh(X.T @ F @ X)
            C = X @ Cp
            Co = C[:, :nocc]
        D = 2.0 * Co @ Co.T
        dv = (B * D).sum((1, 2))
        J = torch.einsum("p,pmn->mn", dv, B)
        H = torch.einsum("pmn,ni->pmi", B, Co)
        K = -torch.einsum("pmi,pni->mn", H, H)
        F0 = h + J + K
        F0 = 0.5 * (F0 + F0.T)
        E = 0.5 * float((D * (h + F0)).sum()) + enuc
        e = X.T @ (F0 @ D @ S - S @ D @ F0) @ X
        err = float(e.abs().max())
        fs, es = (fs + [F0])[-8:], (es + [e])[-8:]
        # to the rounding floor: an error e of the orbitals moves the forces of these nearly dependent sets by far more
        stalled = stalled + 1 if err > 0.5 * best else 0
        if err < 1e-12 or (best < 1e-7 and stalled >= 3):
            break
        best = min(best, err)
        m = len(fs)
        F = F0
        if m > 1:
            Bm = -torch.ones((m + 1, m + 1), dtype=torch.float64)
            Bm[m, m] = 0.0
            for i in range(m):
                for j in range(m):
                    Bm[i, j] = float((es[i] * es[j]).sum())
            Bm[:m, :m] /= Bm[:m, :m].diagonal().max()
            rhs = torch.zeros(m + 1, dtype=torch.float64)
            rhs[m] = -1.0
            co = torch.linalg.solve(Bm, rhs)[:m]
            F = sum(float(c) * f for c, f in zip(co, fs))
    eps, Cp = torch.linalg.eigh(X.T @ F0 @ X)
    Co = (X @ Cp)[:, :nocc]
    D = 2.0 * Co @ Co.T
    Ct = math.sqrt(2.0) * Co
    Wm = 0.5 * D @ F0 @ D
    Bij = torch.einsum("pmn,mi,nj->pij", B, Ct, Ct)
    Xm, c = tri(Lc.T, Bij, True), tri(Lc.T, (B * D).sum((1, 2)), True)
    Y = c[:, None, None] * D - 0.5 * torch.einsum("mi,pij,nj->pmn", Ct, Xm, Ct)
    Zm = torch.outer(c, c) - 0.5 * torch.einsum("pij,qij->pq", Xm, Xm)
    full = torch.zeros(N, dtype=torch.float64, device=x.device)
    full[: len(eps)] = eps
    return np.array([E]), D, full, ex.gradient(x, D, Wm, Y, Zm), Co


def exact(case, seed):
    mols = _molecules(case, seed)
    if sum((_sizes(case, case["n"])[0] * m.natoms // 3) for m in mols) > EXACT_MOST or case["kind"] == "batch":
        return None
    mol = mols[0]
    dev = torch.device("cuda" if torch.cuda.is_available() else "cpu")
    ex = _Exact(mol, case["pure"], dev)
    x = torch.tensor(mol.xyz, dtype=torch.float64, device=dev)
    host = lambda t: t.cpu().numpy()
    if case["kind"] == "integrals":
        S, h, A, T3 = ex.matrices(x)
        return dict(S=host(S), H=host(h), A=host(A), T3=host(T3))
    nocc, tau = mol.nelec // 2, _options(case).get("lindep_tau", 1e-8)
    E, D, eps, g, Co = _solve(ex, x, nocc, tau)
    if case["kind"] == "point":
        # the larger basis: rounding of D alone moves these forces by 1e-4 of their size, here as there
        return dict(energy=E, D=host(D), eps=host(eps), grad=None if case["basis"] == "large" else host(g))
    x1 = torch.tensor(_moved(mol, host(g), int(seed) % 100003), dtype=torch.float64, device=dev)
    E1, _, _, g1, _ = _solve(ex, x1, nocc, tau, Co)
    return [dict(energy=E1, grad=host(g1)), dict(energy=E, grad=host(g))]
