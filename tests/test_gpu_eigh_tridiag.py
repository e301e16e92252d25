"""The tridiagonal eigensolver (orders above 256) on the spectra where its parts can go wrong.

Bounds: a backward-stable FP64 eigensolver has residuals and orthogonality of a few n rounding
units of the norm (n 2.2e-16 = 1e-13 at n = 500); asserted are the 1e-12 / 1e-11 of the random
matrices' test.
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def _matrix(kind, n):
    rng = np.random.default_rng(n)
    if kind == "identity":
        return 2.5 * np.eye(n)
    if kind == "diagonal":
        return np.diag(rng.normal(size=n))
    if kind == "equal blocks":   # uncoupled equal molecules: every eigenvalue repeated
        m = 37
        B = rng.normal(size=(m, m))
        A = np.zeros((n, n))
        for k in range(0, n - m + 1, m):
            A[k:k + m, k:k + m] = (B + B.T) / 2
        return A
    Q, _ = np.linalg.qr(rng.normal(size=(n, n)))
    if kind == "graded":         # an overlap matrix of a nearly dependent basis
        w = np.logspace(-9, 1, n)
    elif kind == "repeated":     # dense, a third of the eigenvalues equal
        w = np.where(np.arange(n) % 3 == 0, 1.0, np.linspace(-2, 2, n))
    else:                        # "clusters": close pairs
        w = np.repeat(np.linspace(-1, 1, (n + 1) // 2), 2)[:n] + 1e-12 * rng.normal(size=n)
    return (Q * w) @ Q.T


@pytest.mark.parametrize("n", [257, 301, 608])
@pytest.mark.parametrize("kind", ["identity", "diagonal", "equal blocks", "graded", "repeated", "clusters"])
def test_special_spectra(kind, n):
    from paper_2407_19614_gb300 import rihf as R
    A = _matrix(kind, n)
    A = (A + A.T) / 2
    W, V = R.eigh(A)
    ref = np.linalg.eigvalsh(A)
    scale = np.abs(ref).max()
    assert np.all(np.diff(W) >= -1e-13 * scale)
    assert np.abs(W - ref).max() <= 1e-12 * scale
    assert np.abs(V.T @ V - np.eye(n)).max() <= 1e-12
    assert np.abs(A @ V - V * W).max() <= 1e-11 * scale
