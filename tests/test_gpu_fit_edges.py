"""The triangular solve of the fit and the DIIS step at the sizes where their kernels change.

The solve takes eight lanes a column up to 64 columns an SM (9728 columns on 152 SMs: N = 139) and
one thread a column above, in 32-row blocks; the sizes here leave remainders of rows (NA mod 32) and
columns (mod 16) on both sides.
"""
import numpy as np
import pytest

from paper_2407_19614_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", ["fp64", "mixed"])
@pytest.mark.parametrize("nwater", [1, 2, 5, 6])
def test_fit_against_lapack(nwater, precision):
    """B = L^{-1} T from the device's own A and T.  The Cholesky factor, and B with it, is defined
    to cond(A) rounding units (first order); B's largest element sets the scale."""
    scipy_linalg = pytest.importorskip("scipy.linalg")
    from paper_2407_19614_gb300 import rihf as R
    ctx = R.Context(W.water_n(nwater, seed=1),
                    precision=R.PRECISION_MIXED if precision == "mixed" else R.PRECISION_FP64)
    A, T, B = ctx.matrix("A"), ctx.matrix("T3"), ctx.matrix("B")
    NA, N = len(A), T.shape[1]
    ref = scipy_linalg.solve_triangular(np.linalg.cholesky(A), T.reshape(NA, -1), lower=True).reshape(T.shape)
    il = np.tril_indices(N)
    err = np.abs(B[:, il[0], il[1]] - ref[:, il[0], il[1]]).max()
    assert err <= np.linalg.cond(A) * 2.2e-16 * np.abs(ref).max()


@pytest.mark.parametrize("size", [3, 5, 16])
def test_diis_history_lengths(size):
    """The converged energy does not depend on the length of the history (3 and 5:
    the ring wraps round; 16: the largest).  conv_e bounds the last step of each."""
    from paper_2407_19614_gb300 import rihf as R
    mol = W.water_monomer(2)
    kw = dict(conv_e=1e-11, conv_diis=1e-8, max_iter=200)
    ref = R.Context(mol, diis_size=8, **kw).scf()["energy"]
    assert abs(R.Context(mol, diis_size=size, **kw).scf()["energy"] - ref) <= 1e-9
