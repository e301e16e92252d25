"""The one-electron lane kernels at every number of lanes a pair, against the warp-cooperative ones.

A basis of s and p shells is the same in Cartesian (x, y, z) and in spherical form (y, z, x), and the two
forms run different kernels.  Clusters of 1, 4, 10, 14 and 20 waters (11 such shells each) get 8, 32, 16, 8 and 4
lanes a pair on 152 SMs, with chunks that end inside a warp.  Integrals to the 1e-12 of the largest
element of the other integral tests.  The forces come from two SCFs whose densities differ by about
conv_diis over the gap (1e-9); a term of the gradient is that times its derivative integrals (below
1e2 in sum), the total is stationary.
"""
import numpy as np
import pytest

from paper_2407_19614_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nwater", [1, 4, 10, 14, 20])
def test_lanes_against_warps(nwater):
    from paper_2407_19614_gb300 import rihf as R
    mol = W.water_n(nwater, 3)
    mol.primary = [s for s in mol.primary if s.l <= 1]
    mol.aux = [s for s in mol.aux if s.l <= 1]
    got = []
    for pure in (1, 0):
        c = R.Context(mol, pure=pure, conv_e=1e-9, conv_diis=1e-9, max_iter=200)
        S, H = c.matrix("S"), c.matrix("H")
        c.scf(guess=5, outputs=False)
        g = c.gradient()
        got.append((S, H, c.matrix("GRAD_PARTS"), g))
        c.close()
    (S, H, P, g), (S0, H0, P0, g0) = got
    at, n = [], 0
    for s in mol.primary:   # spherical positions of the Cartesian functions
        at += [n] if s.l == 0 else [n + 2, n, n + 1]
        n += 2 * s.l + 1
    S, H = S[np.ix_(at, at)], H[np.ix_(at, at)]
    assert np.abs(S - S0).max() <= 1e-12 * np.abs(S0).max()
    assert np.abs(H - H0).max() <= 1e-12 * np.abs(H0).max()
    assert np.abs(P[:2] - P0[:2]).max() <= 1e-7
    assert np.abs(g - g0).max() <= 1e-8
