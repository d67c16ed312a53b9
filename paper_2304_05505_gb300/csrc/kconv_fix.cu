// The FP64 k-mesh convolution (step S3 of the FP64 form) with its DFTs in
// 64-bit fixed point, for meshes whose axes are 1 to 4 points long.
//
//   M^k = IDFT(DFT(D) o Vh) per (P,Q) element (kconv.cu has the conventions)
//
// A radix-2 or radix-4 DFT only adds and subtracts, and a radix-3 one adds two
// products with sqrt(3)/2.  In FP64 that is 1536 operations per element of a
// 4 x 4 x 4 mesh beside the 256 of the product with Vh, and the FP64 pipe does
// 2 per SM and clock: 5.2 ms for N_P = 1200, four fifths of it additions that
// the integer pipe does 30 times as fast.  So each element's N_k values are
// scaled by one power of two to 56-bit integers (2^-56 of the largest; an FP64
// sum rounds at 2^-53), transformed by integer additions that cannot overflow
// (at most 64 terms), turned back to FP64 for the product, and the products
// again scaled and transformed.  Conversions both ways are integer
// operations too (the hardware ones go through the FP64 pipe).
//
// N1 lanes of a warp share an element, lane slot t with the N2 N3 values of
// first mesh index t in registers; the first axis goes across the lanes by
// exchanges with one partner per radix-2 step.  With N1 = 4 the forward
// transform leaves index m = 2 (t & 1) + (t >> 1) in slot t, Vh is read in
// that order, and the inverse starts from it.
//
// Fixed point is no coarser than FP64 here: an FP64 DFT rounds its sums at
// 2^-53 of their size, and every output adds the element's largest input, which
// fixed point rounds at 2^-57 (4 x 4 x 4, rms of the element's largest M: 4e-17
// to 8e-17 against 9e-17 to 1.2e-16 in FP64, for values within one order of
// magnitude to spread over 16 between the k points).  Values with a NaN or an Inf, and products that
// overflow, have no scale: their elements are transformed in FP64.
#include "kconv_dft.cuh"
#include "thc_internal.cuh"

#include <math.h>

namespace {

struct I2 {
  long long x, y;
};

__device__ __forceinline__ I2 operator+(I2 a, I2 b) { return {a.x + b.x, a.y + b.y}; }
__device__ __forceinline__ I2 operator-(I2 a, I2 b) { return {a.x - b.x, a.y - b.y}; }
// i * sign * a
__device__ __forceinline__ I2 turn(I2 a, int sign) { return sign > 0 ? I2{-a.y, a.x} : I2{a.y, -a.x}; }
// sqrt(3)/2 * a (|a| < 2^62): the constant times 2^63, the high word of its product with 2 a
__device__ __forceinline__ long long mul_s3(long long a) { return __mul64hi(2 * a, 7987674492471257551LL); }

// Biased exponent of the larger part.
__device__ __forceinline__ int expo2(double2 v) {
  return max((__double2hiint(v.x) >> 20) & 0x7ff, (__double2hiint(v.y) >> 20) & 0x7ff);
}

// x 2^(56 - e), rounded, with e = E - 1022 and |x| < 2^e.
__device__ __forceinline__ long long to_fixed(double x, int E) {
  const unsigned long long u = (unsigned long long)__double_as_longlong(x);
  const int ex = (int)(u >> 52) & 0x7ff;
  unsigned long long m = (u & 0xfffffffffffffull) | (ex ? 1ull << 52 : 0);
  const int sh = max(ex, 1) - E + 3;
  if (sh >= 0) m <<= min(sh, 4);
  else m = sh > -55 ? (m + (1ull << (-sh - 1))) >> -sh : 0;
  return (long long)u < 0 ? -(long long)m : (long long)m;
}

// m 2^s outside the normal range (out of line: it is as long as the rest).
__device__ __noinline__ double scale_slow(unsigned long long m, int s) { return ldexp((double)m, s); }

// The double nearest v 2^(e - 56).  (Signs are set as bits: a negation goes through the FP64 pipe.)
__device__ __forceinline__ double from_fixed(long long v, int E) {
  unsigned long long m = v < 0 ? -(unsigned long long)v : (unsigned long long)v;
  if (m == 0) return 0.0;
  const int s = __clzll((long long)m) - 1;
  m <<= s;                                       // leading bit 62
  m = (m + 511 + ((m >> 10) & 1)) >> 10;         // 53 bits, to nearest, ties to even
  const int o = E + 7 - s;
  if (o < 1 || o > 2045) {
    const double r = scale_slow(m, E - 1068 - s);
    return v < 0 ? -r : r;
  }
  return __longlong_as_double((long long)(((unsigned long long)(o - 1) << 52) + m | (unsigned long long)v & 1ull << 63));
}

template <int N>
__device__ __forceinline__ void line(I2* x, int step, int sign) {
  if constexpr (N == 2) {
    const I2 a = x[0], b = x[step];
    x[0] = a + b;
    x[step] = a - b;
  } else if constexpr (N == 3) {
    const I2 a = x[0], t = x[step] + x[2 * step], d = x[step] - x[2 * step];
    const I2 m{a.x - (t.x >> 1), a.y - (t.y >> 1)}, s = turn(I2{mul_s3(d.x), mul_s3(d.y)}, sign);
    x[0] = a + t;
    x[step] = m + s;
    x[2 * step] = m - s;
  } else if constexpr (N == 4) {
    const I2 a0 = x[0] + x[2 * step], a1 = x[0] - x[2 * step];
    const I2 b0 = x[step] + x[3 * step], b1 = turn(x[step] - x[3 * step], sign);
    x[0] = a0 + b0;
    x[2 * step] = a0 - b0;
    x[step] = a1 + b1;
    x[3 * step] = a1 - b1;
  }
}

template <int N2, int N3>
__device__ __forceinline__ void planes(I2* x, int sign) {
#pragma unroll
  for (int i = 0; i < N3; i++) line<N2>(x + i, N3, sign);
#pragma unroll
  for (int i = 0; i < N2; i++) line<N3>(x + i * N3, 1, sign);
}

__device__ __forceinline__ I2 swap_xor(I2 v, int m) {
  return {__shfl_xor_sync(0xffffffffu, v.x, m), __shfl_xor_sync(0xffffffffu, v.y, m)};
}
__device__ __forceinline__ I2 from_lane(I2 v, int l) {
  return {__shfl_sync(0xffffffffu, v.x, l), __shfl_sync(0xffffffffu, v.y, l)};
}

// The DFT along the first axis of one value per lane.  inv: from the order the forward one leaves.
template <int N1>
__device__ __forceinline__ I2 across(I2 v, int slot, int el, int sign, bool inv) {
  constexpr int EPW = 32 / N1;
  if constexpr (N1 == 2) {
    const I2 p = swap_xor(v, EPW);
    return slot ? p - v : v + p;
  } else if constexpr (N1 == 3) {
    const int t1 = slot == 2 ? 0 : slot + 1, t2 = slot == 0 ? 2 : slot - 1;
    const I2 p = from_lane(v, min(t1, 2) * EPW + el), q = from_lane(v, min(t2, 2) * EPW + el);
    I2 x[3];                                     // v_0, v_1, v_2
    x[0] = slot == 0 ? v : slot == 1 ? q : p;
    x[1] = slot == 0 ? p : slot == 1 ? v : q;
    x[2] = slot == 0 ? q : slot == 1 ? p : v;
    line<3>(x, 1, sign);
    return slot == 0 ? x[0] : slot == 1 ? x[1] : x[2];
  } else if constexpr (N1 == 4) {
    const int h = slot >> 1, l = slot & 1;
    if (!inv) {
      I2 p = swap_xor(v, 2 * EPW);
      v = h ? p - v : v + p;                     // v_l + v_(l+2), or their difference
      if (h && l) v = turn(v, sign);
      p = swap_xor(v, EPW);
      return l ? p - v : v + p;
    }
    I2 p = swap_xor(v, EPW);
    v = l ? p - v : v + p;
    if (h && l) v = turn(v, sign);
    p = swap_xor(v, 2 * EPW);
    return h ? p - v : v + p;
  } else {
    return v;
  }
}

// The largest e over the lanes that share an element.
template <int N1>
__device__ __forceinline__ int group_max(int e, int el) {
  constexpr int EPW = 32 / N1;
  if constexpr (N1 == 3)
    return max(__shfl_sync(0xffffffffu, e, el), max(__shfl_sync(0xffffffffu, e, EPW + el),
                                                     __shfl_sync(0xffffffffu, e, 2 * EPW + el)));
  if constexpr (N1 >= 2 && N1 != 3) e = max(e, __shfl_xor_sync(0xffffffffu, e, EPW));
  if constexpr (N1 == 4) e = max(e, __shfl_xor_sync(0xffffffffu, e, 2 * EPW));
  return e;
}

// One element by the general FP64 transform, in place in its output (the
// operations of kconv_kernel).
__device__ __noinline__ void general(const double2* D, const double2* Vh, double2* M, long npq, const Twiddles& tw) {
  const int nk = tw.n[0] * tw.n[1] * tw.n[2];
  for (int k = 0; k < nk; k++) M[k * npq] = D[k * npq];
  dft3<double>(M, npq, tw, -1);
  for (int k = 0; k < nk; k++) M[k * npq] = cmul(M[k * npq], Vh[k * npq]);
  dft3<double>(M, npq, tw, +1);
}

template <int N1, int N2, int N3>
__global__ void __launch_bounds__(128) kconv_fix_kernel(const double2* __restrict__ D, const double2* __restrict__ Vh,
                                                        double2* __restrict__ M, long npq,
                                                        const __grid_constant__ Twiddles tw) {
  constexpr int L = N2 * N3, EPW = 32 / N1;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int sl = lane / EPW, el = lane - sl * EPW;
  const bool live = sl < N1;                       // N1 = 3: lanes 30 and 31 idle
  const int slot = live ? sl : 0;
  const long e = ((long)blockIdx.x * 4 + warp) * EPW + el;
  const bool ok = live && e < npq;
  const int ms = N1 == 4 ? 2 * (slot & 1) + (slot >> 1) : slot;
  const double2* d = D + (long)slot * L * npq + e;
  const double2* vh = Vh + (long)ms * L * npq + e;
  double2 in[L];
#pragma unroll
  for (int j = 0; j < L; j++) in[j] = ok ? __ldcs(d + (long)j * npq) : make_double2(0.0, 0.0);
  int E = 0;
#pragma unroll
  for (int j = 0; j < L; j++) E = max(E, expo2(in[j]));
  E = group_max<N1>(E, el);
  I2 x[L];
#pragma unroll
  for (int j = 0; j < L; j++) x[j] = {to_fixed(in[j].x, E), to_fixed(in[j].y, E)};
  // (the kernel's values are on their way while the lanes exchange)
#pragma unroll
  for (int j = 0; j < L; j++) in[j] = ok ? __ldcs(vh + (long)j * npq) : make_double2(0.0, 0.0);
#pragma unroll
  for (int j = 0; j < L; j++) x[j] = across<N1>(x[j], slot, el, -1, false);
  planes<N2, N3>(x, -1);
  int F = 0;
#pragma unroll
  for (int j = 0; j < L; j++) {
    in[j] = cmul(make_double2(from_fixed(x[j].x, E), from_fixed(x[j].y, E)), in[j]);
    F = max(F, expo2(in[j]));
  }
  F = group_max<N1>(F, el);
#pragma unroll
  for (int j = 0; j < L; j++) x[j] = {to_fixed(in[j].x, F), to_fixed(in[j].y, F)};
  planes<N2, N3>(x, +1);
#pragma unroll
  for (int j = 0; j < L; j++) x[j] = across<N1>(x[j], slot, el, +1, true);
  if (!ok) return;
  if (E == 2047 || F == 2047) {   // (the same for all lanes of an element)
    if (slot == 0) general(D + e, Vh + e, M + e, npq, tw);
    return;
  }
  double2* m = M + (long)slot * L * npq + e;
#pragma unroll
  for (int j = 0; j < L; j++) __stcs(m + (long)j * npq, make_double2(from_fixed(x[j].x, F), from_fixed(x[j].y, F)));
}

template <int N1, int N2, int N3>
cudaError_t launch(const double2* D, const double2* Vh, double2* M, long npq, cudaStream_t s) {
  constexpr int EPB = 4 * (32 / N1);
  kconv_fix_kernel<N1, N2, N3><<<(unsigned)((npq + EPB - 1) / EPB), 128, 0, s>>>(D, Vh, M, npq, make_twiddles(N1, N2, N3));
  return cudaGetLastError();
}

template <int N1, int N2>
cudaError_t by_n3(const double2* D, const double2* Vh, double2* M, long npq, int n3, cudaStream_t s) {
  switch (n3) {
    case 1: return launch<N1, N2, 1>(D, Vh, M, npq, s);
    case 2: return launch<N1, N2, 2>(D, Vh, M, npq, s);
    case 3: return launch<N1, N2, 3>(D, Vh, M, npq, s);
    default: return launch<N1, N2, 4>(D, Vh, M, npq, s);
  }
}

template <int N1>
cudaError_t by_n2(const double2* D, const double2* Vh, double2* M, long npq, int n2, int n3, cudaStream_t s) {
  switch (n2) {
    case 1: return by_n3<N1, 1>(D, Vh, M, npq, n3, s);
    case 2: return by_n3<N1, 2>(D, Vh, M, npq, n3, s);
    case 3: return by_n3<N1, 3>(D, Vh, M, npq, n3, s);
    default: return by_n3<N1, 4>(D, Vh, M, npq, n3, s);
  }
}

}  // namespace

bool kconv_fix_applies(int n1, int n2, int n3) { return n1 <= 4 && n2 <= 4 && n3 <= 4; }

cudaError_t kconv_fix_z(const double2* D, const double2* Vh, double2* M, long npq, int n1, int n2, int n3,
                        cudaStream_t s) {
  switch (n1) {
    case 1: return by_n2<1>(D, Vh, M, npq, n2, n3, s);
    case 2: return by_n2<2>(D, Vh, M, npq, n2, n3, s);
    case 3: return by_n2<3>(D, Vh, M, npq, n2, n3, s);
    default: return by_n2<4>(D, Vh, M, npq, n2, n3, s);
  }
}
