// Cholesky factor of a real symmetric matrix and the inverse of the factor (chol.cu).
#pragma once

#include "oz_gemm.cuh"

// L (n x n, row-major, lower, zero above the diagonal) with S = L L^T, in FP64.
// A pivot that is not above 1e-12 S_jj sets *bad (L is then unusable).
cudaError_t chol_factor(const double* S, double* L, int n, int* bad, cudaStream_t s);

// Linv = L^-1 (same form).  T: scratch of n x n doubles; w: scratch of the products of the large blocks.
cudaError_t chol_inverse(const double* L, double* Linv, double* T, int n, const OzWork& w, cudaStream_t s);

// X = (L L^T)^-1 X for the columns of X[n][ldx], as L^-T (L^-1 X).  Y: scratch of n x ldx doubles.
cudaError_t chol_apply(const double* Linv, double* X, double* Y, int n, int ldx, const OzWork& w, cudaStream_t s);
