// Cholesky factor of a real symmetric matrix (chol.cu).
#pragma once

#include <cuda_runtime.h>

// L (n x n, row-major, lower, zero above the diagonal) with S = L L^T, in FP64.
// A pivot that is not above 1e-12 S_jj sets *bad (L is then unusable).
cudaError_t chol_factor(const double* S, double* L, int n, int* bad, cudaStream_t s);
