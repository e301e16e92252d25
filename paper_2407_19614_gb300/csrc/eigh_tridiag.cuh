// Symmetric eigen-decomposition through the tridiagonal form (eigh_tridiag.cu).
#pragma once
#include "linalg.cuh"

namespace rihf {

// Eigenvalues lam (unsorted) and eigenvectors V (column k belongs to lam[k]) of
// the n x n symmetric FP64 matrix A, to FP64 accuracy relative to its norm; ws:
// tridiag_workspace(n) doubles.  la.flag[1] is set when a grid barrier ran out of
// time (2 s).
void tridiag_eigh(const LaCtx& la, const double* A, int n, double* lam, double* V, double* ws);

}  // namespace rihf
