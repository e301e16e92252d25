"""The digit-plane GEMM over its column tiles and the slicing over its chunk splits.

Sizes sit on both sides of each rule: 16 or 32 columns a tile while that leaves no more than one
tile an SM, 48 for 65..96 columns, 64 otherwise; ragged last tiles of rows, columns and K; rows of
odd length (element loads) and of multiples of 8 (16-byte loads); K blocks of one chunk, of a few
and of more than the 16 that stay in registers.  Bound: that of the plain GEMM's tests, and what the
fixed-point sums drop at each read-out (every 128 to 256 elements): the two lowest of the seven
anti-diagonals are shifted down, and each loses less than one unit, 2^-49 of the product of the two
rows' leading powers of two.
"""
import numpy as np
import pytest

from test_gpu_tc_gemm import _bound, _case

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("M,N,K,kblock", [
    (1, 1, 1, 0), (129, 17, 33, 0), (384, 384, 384, 0), (2000, 200, 40, 0), (1300, 470, 72, 0), (4000, 300, 64, 0),
    (20000, 80, 41, 0), (20000, 96, 64, 0), (20000, 100, 96, 0), (20000, 50, 8, 0), (20000, 30, 7, 0),
    (300, 70, 1999, 60), (140, 130, 2000, 20), (200, 40, 672, 0)])
@pytest.mark.parametrize("digits", [4, 5, 6, 7])
def test_tiles(M, N, K, kblock, digits):
    from paper_2407_19614_gb300 import rihf
    A, B = _case(M, N, K, seed=M + N + K, wide=True)
    C = rihf.tc_dgemm(A, B, digits=digits, kblock=kblock)
    readouts = -(-K // 128) + (-(-K // (32 * kblock)) if kblock else 0)
    dropped = 2 * 2.0 ** -49 * readouts * np.outer(np.abs(A).max(axis=1), np.abs(B).max(axis=1))
    assert np.all(np.abs(C - A @ B.T) <= _bound(A, B, digits, kblock) + dropped)
