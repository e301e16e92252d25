"""The eigensolver over the norm of its matrix.

Scaling by a power of two changes no rounding, so the bounds are those of the random matrices at
norm 1 (a few n rounding units of the norm), relative to the norm.  The orders take both forms of the
FP32 Jacobi (one CTA up to 64, a cluster above), whose FP32 start reaches from 1e-36 to 1e36, and the
tridiagonal path above 256, whose refinement squares entries in FP64.
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def _check(n, scale):
    from paper_2407_19614_gb300 import rihf as R
    M = np.random.default_rng(n).normal(size=(n, n))
    A = (M + M.T) / 2
    A /= np.abs(np.linalg.eigvalsh(A)).max()
    W, V = R.eigh(A * scale)
    W /= scale
    assert np.abs(W - np.linalg.eigvalsh(A)).max() <= 1e-12
    assert np.abs(V.T @ V - np.eye(n)).max() <= 1e-12
    assert np.abs(A @ V - V * W).max() <= 1e-11


@pytest.mark.parametrize("n", [24, 64, 65, 200])
@pytest.mark.parametrize("scale", [1e-35, 1e-20, 1e-14, 1e-11, 1e12, 1e20, 1e35])
def test_jacobi_norms(n, scale):
    _check(n, scale)


@pytest.mark.parametrize("n", [257, 400])
@pytest.mark.parametrize("scale", [1e-140, 1e-60, 1e-36, 1e-20, 1e20, 1e36, 1e140])
def test_tridiagonal_norms(n, scale):
    _check(n, scale)
