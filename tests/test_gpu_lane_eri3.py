"""The one-lane-per-task integral kernels at the edges of their classes and ranges, against the oracle.

Integrals element-wise to 1e-12 of the largest element (the bound of the other integral tests: sums of a
few hundred FP64 terms, each a few rounding units).  Gradients to the 1e-8 Eh/bohr of the other
parity tests, in a basis whose overlap is well conditioned: an orbital error e moves the forces by
about e / (gap sqrt(lambda_min(S))), so SCF errors of 1e-9 stay below 1e-8 at lambda_min 0.017 (the
workloads' nearly dependent f/g set has lambda_min ~ 1e-7 and moves them by 1e-8 to 1e-6).
"""
import copy

import numpy as np
import pytest

from oracle import rihf as O
from paper_2407_19614_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def _R():
    from paper_2407_19614_gb300 import rihf as R
    R.load()
    return R


def _shuffled(mol, seed):
    """Shells in random order: pairs with la < lb, equal l on either side, atoms interleaved."""
    rng = np.random.default_rng(seed)
    mol.primary = [mol.primary[i] for i in rng.permutation(len(mol.primary))]
    mol.aux = [mol.aux[i] for i in rng.permutation(len(mol.aux))]
    return mol


def _mixed_contraction(mol):
    """Contraction lengths 1..3 within one class (lanes of a warp with different loop counts)."""
    for i, s in enumerate(mol.primary):
        k = 1 + i % 3
        s.exps, s.coefs = [s.exps[0] * f for f in (1.0, 0.6, 2.3)[:k]], [0.5, 0.4, 0.2][:k]
    for i, s in enumerate(mol.aux):
        k = 1 + i % 2
        s.exps, s.coefs = [s.exps[0] * f for f in (1.0, 1.7)[:k]], [0.6, 0.5][:k]
    return mol


def _conditioned(seed):
    """s to f primary and s to g auxiliary shells, one or two per l: every class, lambda_min(S) = 0.017."""
    mol = W.water_n(1, seed)
    prim = {8: [(0, 0.35), (0, 1.9), (1, 0.5), (2, 0.9), (3, 1.3)], 1: [(0, 0.45), (1, 0.9)]}
    aux = {8: [(0, 0.5), (0, 1.6), (0, 5.0), (1, 0.7), (1, 2.5), (2, 0.9), (2, 3.0), (3, 1.1), (4, 1.4)],
           1: [(0, 0.5), (0, 1.8), (1, 0.9), (2, 1.2)]}
    mol.primary = [W.Shell(a, l, [x], [1.0]) for a, z in enumerate(mol.Z) for l, x in prim[int(z)]]
    mol.aux = [W.Shell(a, l, [x], [1.0]) for a, z in enumerate(mol.Z) for l, x in aux[int(z)]]
    return mol


def _two_f_atoms():
    """Two waters with one f shell each, 3.6 bohr apart: (f f| pairs over two atoms (overlap up to 0.18,
    density 4e-3: their derivatives are 1e5 times the bound), lambda_min(S) = 0.059."""
    mol = W.water_n(2, 7)
    d = mol.xyz[3] - mol.xyz[0]
    mol.xyz = mol.xyz.copy()
    mol.xyz[3:] -= d * (1.0 - 3.6 / np.linalg.norm(d))
    prim = {8: [(0, 0.35), (0, 1.9), (1, 0.5), (2, 0.9), (3, 0.5)], 1: [(0, 0.45)]}
    aux = {8: [(0, 0.5), (0, 1.6), (0, 5.0), (1, 0.7), (1, 2.5), (2, 0.9), (2, 3.0), (3, 1.1), (4, 1.4)],
           1: [(0, 0.5), (0, 1.8), (1, 0.9), (2, 1.2)]}
    mol.primary = [W.Shell(a, l, [x], [1.0]) for a, z in enumerate(mol.Z) for l, x in prim[int(z)]]
    mol.aux = [W.Shell(a, l, [x], [1.0]) for a, z in enumerate(mol.Z) for l, x in aux[int(z)]]
    return mol


def _case(name):
    if name == "f on two atoms":
        return _shuffled(_two_f_atoms(), 7)
    if name == "f and g conditioned":
        return _shuffled(_conditioned(5), 5)
    if name == "mixed contraction conditioned":
        return _mixed_contraction(_shuffled(_conditioned(6), 6))
    if name == "small shuffled":
        return _shuffled(W.water_n(2, 1), 1)
    if name == "f and g shuffled":
        return _shuffled(W.water_n(1, 2, "large"), 2)
    if name == "mixed contraction":
        return _mixed_contraction(_shuffled(W.water_n(1, 3, "large"), 3))
    mol = W.water_n(2, 4, "large" if name == "far, f and g" else "small")
    mol.xyz = mol.xyz.copy()
    # Boys arguments on both sides of the table's end (T = 40) and of the exponential's cut (T = 72)
    mol.xyz[3:] += np.array([0.0, 0.0, 6.0 if name == "middle distance" else 25.0])
    return mol


@pytest.mark.parametrize("name", ["small shuffled", "f and g shuffled", "mixed contraction", "middle distance",
                                  "far, f and g"])
def test_three_centre_integrals(name):
    R = _R()
    mol = _case(name)
    s = O.System(mol)
    ctx = R.Context(mol)
    T = ctx.matrix("T3")
    ctx.close()
    assert np.abs(T - s.T3).max() <= 1e-12 * np.abs(s.T3).max()


@pytest.mark.parametrize("name", ["small shuffled", "f and g shuffled", "mixed contraction", "far, f and g"])
def test_metric_and_one_electron(name):
    R = _R()
    mol = _case(name)
    s = O.System(mol)
    ctx = R.Context(mol)
    for what, ref in (("A", s.A), ("S", s.S), ("H", s.h)):
        assert np.abs(ctx.matrix(what) - ref).max() <= 1e-12 * np.abs(ref).max(), what
    ctx.close()


@pytest.mark.parametrize("name", ["small shuffled", "f and g conditioned", "mixed contraction conditioned",
                                  "middle distance", "f on two atoms"])
def test_three_centre_derivatives(name):
    R = _R()
    mol = _case(name)
    s = O.System(mol)
    r = O.rihf_energy(s, conv_e=1e-12, conv_diis=1e-9)
    ref = O.rihf_gradient_terms(s, r).grad
    ctx = R.Context(mol, conv_e=1e-10, conv_diis=1e-8, max_iter=100)
    ctx.scf(guess=0, outputs=False)
    g = ctx.gradient()
    ctx.close()
    assert np.abs(g - ref).max() <= 1e-8
    assert np.abs(g.sum(0)).max() <= 1e-9


def test_batch_of_spherical_and_cartesian_members():
    """One batched step over contexts of both bases equals the members run alone."""
    R = _R()
    mols = [W.water_n(n, 10 + n) for n in (2, 1, 3)]
    kw = dict(conv_e=1e-10, conv_diis=1e-9, max_iter=100)
    pure = [1, 0, 1]
    ctx = [R.Context(copy.deepcopy(m), pure=p, **kw) for m, p in zip(mols, pure)]
    E, grads, _ = R.batch_step(ctx, [m.xyz for m in mols], guess=0)
    for c in ctx:
        c.close()
    for m, p, e, g in zip(mols, pure, E, grads):
        c = R.Context(m, pure=p, **kw)
        assert abs(c.scf(guess=0, outputs=False)["energy"] - e) <= 1e-9
        assert np.abs(c.gradient() - g).max() <= 1e-8
        c.close()
