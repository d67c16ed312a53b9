// Blocked Cholesky factorisation in FP64.
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
// The solve is a forward and a backward substitution per right-hand side
// (chol_solve, isdf_common.cuh).  Two products with the inverse of L from
// digits took 4 ms in place of 70 at n = 600 and 64000 right-hand sides, but
// are not its equal: a row of L^-1 carries 1 / d_j and a column of the
// right-hand sides d_j, d_j the scale of point j, so that rounding either at
// 2^-63 of its largest entry loses the points of low density (xi 1e-9 of its
// largest entry for densities 1e8 apart, where substitution keeps 2e-15), and
// the inverse itself is not backward stable.
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
