// Blocked Cholesky factorisation in FP64, the inverse of the factor, and the
// solve with many right-hand sides as two matrix products.
//
// The factor: right-looking in panels of 32 columns.  One warp factors the
// diagonal block (a row per lane, in registers), the rows below follow by
// substitution (a row per thread), and the trailing block is updated in
// 16 x 16 tiles, small so that the FP64 pipe of every SM (2 multiply-adds a
// clock) has work.  Every element still goes through the multiply-adds of the
// column-by-column algorithm in the same order, so the bits of L are those
// of chol_column's left-looking sums, which every thread redid from column 0
// for each of the n dependent launches (34 ms at n = 600, 134 ms at n = 1200).
//
// The inverse: [A 0; B C]^-1 = [A^-1 0; -C^-1 B A^-1 C^-1] from the inverted
// diagonal blocks of 32 upward, all pairs of a level in one launch, the
// levels of 256 rows and more on the tensor cores.
//
// The solve: L^-T (L^-1 X), both products on the tensor cores
// (oz_gemm.cu), in place of one substitution per thread and right-hand side,
// which runs at the rate of the FP64 pipe.
#include "chol.cuh"

#include <algorithm>

namespace {

constexpr int CB = 32;

// L = lower part of S, the rest zero.
__global__ void __launch_bounds__(256) chol_init(const double* __restrict__ S, double* __restrict__ L, int n) {
  const long i = (long)blockIdx.x * 256 + threadIdx.x;
  if (i >= (long)n * n) return;
  const int r = (int)(i / n), c = (int)(i % n);
  L[i] = c <= r ? S[i] : 0.0;
}

// The factor of the diagonal block at j0, in place.  One warp, lane = row.
__global__ void __launch_bounds__(CB) chol_diag(const double* __restrict__ S, double* __restrict__ L, int n, int j0,
                                                int* bad) {
  const int i = threadIdx.x, m = min(CB, n - j0);
  double a[CB];
#pragma unroll
  for (int j = 0; j < CB; j++) a[j] = i < m && j <= i ? L[(long)(j0 + i) * n + j0 + j] : (j == i ? 1.0 : 0.0);
  const double sd = i < m ? S[(long)(j0 + i) * n + j0 + i] : 1.0;
  bool ok = true;
#pragma unroll
  for (int j = 0; j < CB; j++) {
    const double d = __shfl_sync(0xffffffffu, a[j], j);
    ok = ok && d > 1e-12 * __shfl_sync(0xffffffffu, sd, j);
    const double l = sqrt(d);
    a[j] = i == j ? l : a[j] / l;
#pragma unroll
    for (int k = j + 1; k < CB; k++) a[k] = fma(-a[j], __shfl_sync(0xffffffffu, a[j], k), a[k]);
  }
  if (!ok && i == 0) atomicOr(bad, 1);
#pragma unroll
  for (int j = 0; j < CB; j++)
    if (j <= i && i < m) L[(long)(j0 + i) * n + j0 + j] = a[j];
}

// Rows below the diagonal block, by substitution: a row per thread.
__global__ void __launch_bounds__(CB) chol_panel(double* __restrict__ L, int n, int j0) {
  __shared__ double d[CB][CB + 1], a[CB][CB + 1];
  const int t = threadIdx.x, i0 = j0 + CB + blockIdx.x * CB, rows = min(CB, n - i0);
  for (int r = 0; r < CB; r++) {
    d[r][t] = L[(long)(j0 + r) * n + j0 + t];
    if (r < rows) a[r][t] = L[(long)(i0 + r) * n + j0 + t];
  }
  __syncwarp();
  if (t < rows) {
    double x[CB];
#pragma unroll
    for (int j = 0; j < CB; j++) {
      double v = a[t][j];
#pragma unroll
      for (int q = 0; q < j; q++) v = fma(-x[q], d[j][q], v);
      x[j] = v / d[j][j];
    }
#pragma unroll
    for (int j = 0; j < CB; j++) a[t][j] = x[j];
  }
  __syncwarp();
  for (int r = 0; r < rows; r++) L[(long)(i0 + r) * n + j0 + t] = a[r][t];
}

// The inverses of the diagonal blocks (a block each, column per lane); Linv is zero elsewhere.
__global__ void __launch_bounds__(CB) inv_diag(const double* __restrict__ L, double* __restrict__ Linv, int n) {
  __shared__ double d[CB][CB + 1];
  const int i = threadIdx.x, j0 = blockIdx.x * CB, m = min(CB, n - j0);
  for (int r = 0; r < CB; r++)
    d[r][i] = r < m && i <= r ? L[(long)(j0 + r) * n + j0 + i] : (r == i ? 1.0 : 0.0);
  __syncwarp();
  double x[CB];
#pragma unroll
  for (int r = 0; r < CB; r++) {
    double v = r == i ? 1.0 : 0.0;
#pragma unroll
    for (int t = 0; t < r; t++) v -= d[r][t] * x[t];
    x[r] = v / d[r][r];
  }
#pragma unroll
  for (int r = 0; r < CB; r++)
    if (i <= r && r < m) Linv[(long)(j0 + r) * n + j0 + i] = x[r];
}

// Trailing update L[i][k] -= sum_t L[i][j0 + t] L[k][j0 + t], i >= k >= j0 + 32, 16 x 16 tiles.
__global__ void __launch_bounds__(256) chol_update(double* __restrict__ L, int n, int j0) {
  __shared__ double sa[16][CB + 1], sb[16][CB + 1];
  if (blockIdx.x > blockIdx.y) return;
  const int k0 = j0 + CB + blockIdx.x * 16, i0 = j0 + CB + blockIdx.y * 16;
  for (int q = threadIdx.x; q < 16 * CB; q += 256) {
    const int r = q / CB, t = q % CB;
    sa[r][t] = i0 + r < n ? L[(long)(i0 + r) * n + j0 + t] : 0.0;
    sb[r][t] = k0 + r < n ? L[(long)(k0 + r) * n + j0 + t] : 0.0;
  }
  __syncthreads();
  const int k = threadIdx.x & 15, i = threadIdx.x >> 4;
  if (i0 + i >= n || k0 + k > i0 + i) return;
  double v = L[(long)(i0 + i) * n + k0 + k];
#pragma unroll
  for (int t = 0; t < CB; t++) v = fma(-sa[i][t], sb[k][t], v);
  L[(long)(i0 + i) * n + k0 + k] = v;
}

// C = alpha A B for the pairs of one level of the inverse (blockIdx.z = pair), 16 x 16 tiles.  step 0: T = B Ainv
// (the pair's lower left block of L with the inverse above it); step 1: Linv's block = -Cinv T.
__global__ void __launch_bounds__(256) inv_level(const double* __restrict__ L, double* __restrict__ Linv,
                                                 double* __restrict__ T, int n, int h, int step) {
  __shared__ double sa[16][17], sb[16][17];
  const int c0 = 2 * h * blockIdx.z, r0 = c0 + h, rows = min(h, n - r0);
  const int m0 = blockIdx.y * 16, n0 = blockIdx.x * 16, x = threadIdx.x & 15, y = threadIdx.x >> 4;
  if (m0 >= rows || n0 >= h) return;
  const int K = step ? rows : h;
  double v = 0.0;
  for (int k0 = 0; k0 < K; k0 += 16) {
    const bool ia = m0 + y < rows && k0 + x < K, ib = k0 + y < K && n0 + x < h;
    sa[y][x] = ia ? (step ? Linv[(long)(r0 + m0 + y) * n + r0 + k0 + x] : L[(long)(r0 + m0 + y) * n + c0 + k0 + x])
                  : 0.0;
    sb[y][x] = ib ? (step ? T[(long)(r0 + k0 + y) * n + c0 + n0 + x] : Linv[(long)(c0 + k0 + y) * n + c0 + n0 + x])
                  : 0.0;
    __syncthreads();
#pragma unroll
    for (int t = 0; t < 16; t++) v += sa[y][t] * sb[t][x];
    __syncthreads();
  }
  if (m0 + y < rows && n0 + x < h) {
    const long o = (long)(r0 + m0 + y) * n + c0 + n0 + x;
    if (step) Linv[o] = -v;
    else T[o] = v;
  }
}

}  // namespace

cudaError_t chol_factor(const double* S, double* L, int n, int* bad, cudaStream_t s) {
  chol_init<<<(unsigned)(((long)n * n + 255) / 256), 256, 0, s>>>(S, L, n);
  for (int j = 0; j < n; j += CB) {
    chol_diag<<<1, CB, 0, s>>>(S, L, n, j, bad);
    const int below = n - j - CB;
    if (below <= 0) break;
    chol_panel<<<(below + CB - 1) / CB, CB, 0, s>>>(L, n, j);
    const unsigned t = (unsigned)((below + 15) / 16);
    chol_update<<<dim3(t, t), 256, 0, s>>>(L, n, j);
  }
  return cudaGetLastError();
}

cudaError_t chol_inverse(const double* L, double* Linv, double* T, int n, const OzWork& w, cudaStream_t s) {
  cudaError_t e0 = cudaMemsetAsync(Linv, 0, sizeof(double) * (size_t)n * n, s);
  if (e0 != cudaSuccess) return e0;
  inv_diag<<<(n + CB - 1) / CB, CB, 0, s>>>(L, Linv, n);
  for (int h = CB; h < n; h *= 2) {
    const int pairs = (n - h + 2 * h - 1) / (2 * h);
    if (h < 256) {
      const unsigned t = (unsigned)((h + 15) / 16);
      for (int step = 0; step < 2; step++) inv_level<<<dim3(t, t, pairs), 256, 0, s>>>(L, Linv, T, n, h, step);
      continue;
    }
    for (int p = 0; p < pairs; p++) {
      const long c0 = 2L * h * p, r0 = c0 + h;
      const int rows = std::min(h, (int)(n - r0));
      cudaError_t e = oz_gemm_d(false, true, rows, h, h, L + r0 * n + c0, n, Linv + c0 * n + c0, n, T + r0 * n + c0, n,
                                1.0, false, w, s);
      if (e == cudaSuccess)
        e = oz_gemm_d(false, true, rows, h, rows, Linv + r0 * n + r0, n, T + r0 * n + c0, n, Linv + r0 * n + c0, n,
                      -1.0, false, w, s);
      if (e != cudaSuccess) return e;
    }
  }
  return cudaGetLastError();
}

cudaError_t chol_apply(const double* Linv, double* X, double* Y, int n, int ldx, const OzWork& w, cudaStream_t s) {
  cudaError_t e = oz_gemm_d(false, true, n, ldx, n, Linv, n, X, ldx, Y, ldx, 1.0, false, w, s);
  if (e != cudaSuccess) return e;
  return oz_gemm_d(true, true, n, ldx, n, Linv, n, Y, ldx, X, ldx, 1.0, false, w, s);
}
