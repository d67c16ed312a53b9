// FP64 matrix products on the tensor cores from exact bf16 digits (oz_gemm.cu).
#pragma once

#include "thc_internal.cuh"

// Deepest real K of a product (its int64 sums stay below 2^62).
constexpr long OZ_MAX_K = 1L << 19;

// Scratch bytes for a product of this shape taken whole (complex), and the
// least a product of depth K (complex) can run with.
size_t oz_work_bytes(int M, int N, int K, int batch);
size_t oz_work_min(int K);

// Whether w has room for the digits of this product (complex, or real), whole
// or in slabs.
bool oz_fits(int M, int N, int K, int batch, bool real, const OzWork& w);

// Test hooks: the most scratch that products on the calling thread use from now
// on (negative: all they have), and the slabs of a product with `bytes` of it:
// batch entries, rows of A and rows of B of a slab; false where none fits.
void oz_limit(long long bytes);
bool oz_plan(int M, int N, int K, int batch, bool real, size_t bytes, int plan[3]);

// Allocates scratch: `want` bytes, or halves of it and at last `least` where the
// device has no room for more (cudaErrorMemoryAllocation when it has not even
// that), and clears its error word on `s`.  oz_free gives it back.
cudaError_t oz_alloc(OzWork& w, size_t want, size_t least, cudaStream_t s);
void oz_free(OzWork& w);

// Whether the digit form is the faster one for this complex product.
bool oz_wins(int M, int N, int K, int batch);

// gemm_z's product in the faster of its two forms (w.buf may be null).
cudaError_t gemm_z_best(int la, int lb, int M, int N, int K, const double2* A, int lda, long sA, const double2* B,
                        int ldb, long sB, double2* C, int ldc, long sC, int batch, const OzWork& w, cudaStream_t s);

// gemm_z's product (operand layouts of GemmA, GemmB) from digits.  check: to
// FP64 accuracy of every entry (those that seven digits relative to the rows'
// largest entries do not hold to it are computed with eight or in FP64); else to 4 K 2^-62 of the
// product of the largest entries of its two rows.
cudaError_t oz_gemm_z(int la, int lb, int M, int N, int K, const double2* A, int lda, long sA, const double2* B,
                      int ldb, long sB, double2* C, int ldc, long sC, int batch, bool check, const OzWork& w,
                      cudaStream_t s);

// The unchecked product of A (any layout) with a B of N columns stored [k][n]
// whose digits were prepared once: oz_lane_bytes of device memory at `lanes`.
size_t oz_lane_bytes(int N, int K);
size_t oz_lanes_work(int M, int K);                  // scratch for the digits of A (M rows)
bool oz_lanes_fit(int M, int K, const OzWork& w);    // w has that much
cudaError_t oz_lane_prepare(const double2* B, int ldb, int N, int K, void* lanes, cudaStream_t s);
cudaError_t oz_gemm_z_lanes(int la, int M, int N, int K, const double2* A, int lda, void* lanes, double2* C, int ldc,
                            const OzWork& w, cudaStream_t s);

// Real C[m][n] = alpha sum_k A(m, k) B(n, k) (+ C when acc): A(m, k) = A[m lda + k]
// or, a_km, A[k lda + m]; B(n, k) = B[n ldb + k] or, b_kn, B[k ldb + n].  alpha is 1 or -1.
// check as in oz_gemm_z (2 K 2^-62).
cudaError_t oz_gemm_d(bool a_km, bool b_kn, int M, int N, int K, const double* A, long lda, const double* B, long ldb,
                      double* C, long ldc, double alpha, bool acc, bool check, const OzWork& w, cudaStream_t s);
