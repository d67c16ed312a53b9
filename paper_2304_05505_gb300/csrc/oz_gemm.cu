// FP64 matrix products on the tensor cores (tcgen05, sm_103a) from exact
// digits: the error-free splitting of Ozaki, Ogita, Oishi and Rump (2012).
//
// The GB300's FP64 pipe is 1.25 TFLOP/s for the whole device, 1/1500 of its
// bf16 tensor rate.  Every operand row is scaled by a power of two and written
// in seven balanced digits of radix 512,
//   x = 2^(e - 8) (d_0 + 2^-9 d_1 + ... + 2^-54 d_6),  d_s in [-256, 256],
// 2^e above the row's largest entry (62 bits of the row scale, against the 53
// of a double).  A digit has at most 8 significant bits, so the planes
// 2^(-9 s) d_s are exact bf16 numbers, products of two digits are exact in
// FP32, and with C_c = sum over s + t = c of A_s B_t
//   A B = 2^(e_a + e_b - 16) (C_0 + C_1 + ... + C_7)   (C_8 and on dropped, 2^-72:
// C_7 costs 6 of the 34 digit products; without it rows with a few dominant
// entries, as those of the collocation, lose 1e-15 of their products).
// Over a chunk of 64 K the classes C_0 .. C_3 are sums of at most 4 x 64
// integers of at most 2^16 in units of 2^(-9 c): below 2^24, where the tensor
// core's FP32 accumulator is exact whatever its rounding.  After every chunk
// they are added into one int64 per output (units of C_3; |sum| < K 2^43), with
// the whole units of C_4; what is left of C_4 and C_5 + C_6 + C_7 go into one FP32
// number.  The double is rounded once, from integers.  So the result carries
// the error of rounding the operands at 2^-63 of their row scale, the dropped
// classes and one final rounding: 5e-17 of the result on random operands of
// any depth, where the FP64 kernel's running sums leave 4e-16 (K = 60) to
// 3e-15 (K = 3840).
//
// Complex products run as real ones with K = 2 K: one operand plain
// (interleaved), the smaller one embedded as rows (re, -im) and (im, re).
//
// One CTA per SM loops over 128 x 80 output tiles, all of K each:
//   warp 0    TMA: one box of [7 planes][128 rows][32 K] and one of
//             [7][80][32] per stage (91 KB, two stages, 64B swizzle)
//   warp 1    34 digit products per 16 K, one MMA (128 x 80 x 16) each, into
//             six accumulators of 80 TMEM columns: C_0 .. C_4, and C_5 + C_6 + C_7.
//             A wider tile would read less shared memory per product (6.5 KB
//             here, 52 cycles of 40 MMA cycles), but six accumulators fill
//             TMEM: C_4 shares none, since rounding it with C_5 .. C_7 on
//             the way would leave 2^-51 of the result.
//   warps 4-19  drain one accumulator after the other, each as soon as the
//             chunk's last product into it is done and while the later classes
//             are still being multiplied; the next chunk starts on C_0 when C_0
//             is drained.  So the accumulators need no second set.
// The integer epilogue keeps the FP64 pipe (2 results per SM and clock) out of
// the kernel: conversion and rounding of an output are about 30 integer
// instructions.
#include "oz_gemm.cuh"
#include "mbarrier.cuh"

#include <cuda.h>
#include <cudaTypedefs.h>

#include <algorithm>

namespace {

constexpr int ND = 7;                                  // digits
constexpr int TL = 128, TN = 80, TK = 32;              // lane rows, column rows, K of a stage
constexpr uint32_t LPL = TL * TK * 2, CPL = TN * TK * 2;    // bytes of a plane tile: 8 KB, 5 KB
constexpr uint32_t STAGE = ND * (LPL + CPL);           // 91 KB
constexpr int NACC = 6;                                // accumulators: C_0 .. C_4, and C_5 + C_6 + C_7
constexpr int STAGES = 2;
constexpr int CHUNK_ST = 2;                            // stages of an exact chunk (64 K)
constexpr size_t SMEM = STAGES * STAGE + 1024 + 128;
constexpr int EPI0 = 4, EPI_W = 16, NT = 32 * (EPI0 + EPI_W);
constexpr int EC = TN / 4;                             // columns of an epilogue warp
constexpr int NB_ROW = 2047;                           // biased exponent of a row with a NaN or an Inf
constexpr size_t HEAD = 1024;                          // bytes before the planes: the error block

static_assert(SMEM <= 232448, "227 KB of shared memory per block");

struct OzMaps {
  CUtensorMap l, n;
};

struct OzShape {
  int nl, nn;        // valid lanes (rows of the lane operand) and columns
  int nst;           // K stages
  int tl, tn;        // tiles
  int lsh, nsh;      // exponent index = row >> sh (embedded operands: pairs of rows share one)
  long el, en;       // exponents per batch entry
  long units;
  int pairs;         // columns 2m, 2m + 1 are the real and imaginary part of output row m
  int acc;           // add to out
  double alpha;
  long ldo, sbo;     // doubles (pairs: double2)
};

__device__ __forceinline__ void mma_bf16(uint32_t d, uint64_t a, uint64_t b, uint32_t accumulate) {
  // kind::f16, D f32 (bit 4), A and B bf16 (bits 7 and 10), K-major, N >> 3 at bit 17, M >> 4 at bit 24
  constexpr uint32_t idesc =
      (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(TN >> 3) << 17) | ((uint32_t)(TL >> 4) << 24);
  asm volatile(
      "{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n"
      " tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}" ::"r"(d),
      "l"(a), "l"(b), "r"(idesc), "r"(accumulate)
      : "memory");
}

__device__ __forceinline__ void commit(uint32_t bar) {
  asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(bar) : "memory");
}

__device__ __forceinline__ void tc_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }

// K-major tile, 64B swizzle, 8-row groups 512 B apart (see tc_gemm.cu).
__device__ __forceinline__ uint64_t desc64(uint32_t addr) {
  return (uint64_t)((addr & 0x3FFFF) >> 4) | ((uint64_t)1 << 16) | ((uint64_t)(512 >> 4) << 32) | ((uint64_t)1 << 46) |
         ((uint64_t)4 << 61);
}

// 10 consecutive columns of this thread's TMEM lane (half of an epilogue warp's: registers).
constexpr int EH = EC / 2;
static_assert(EH == 10, "tmem_ld10");
__device__ __forceinline__ void tmem_ld10(uint32_t t, float* v) {
  uint32_t r[10];
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%10];\n"
      "tcgen05.ld.sync.aligned.32x32b.x2.b32 {%8, %9}, [%11];\n"
      "tcgen05.wait::ld.sync.aligned;"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]),
        "=r"(r[9])
      : "r"(t), "r"(t + 8)
      : "memory");
#pragma unroll
  for (int i = 0; i < 10; i++) v[i] = __uint_as_float(r[i]);
}

// v 2^s outside the normal range (out of line: it is as long as the rest).
__device__ __noinline__ double scale_slow(double v, int s) { return ldexp(v, s); }

// The double nearest (a + f) 2^sexp (a an integer, |a| < 2^62, f a small FP32 part), by integer operations
// (a negation, too, would go through the FP64 pipe).
__device__ __forceinline__ double round_sum(long long a, float f, int sexp) {
  const int fi = __float2int_rn(f);          // |f| < 2^22: at most 2^8 per chunk of 64 K
  a += fi;
  f -= (float)fi;                            // |f| <= 1/2
  unsigned long long m = a < 0 ? -(unsigned long long)a : (unsigned long long)a;
  if (m == 0) return f == 0.f ? 0.0 : scale_slow((double)f, sexp);
  if (a < 0) f = -f;
  int s = __clzll((long long)m) - 1;
  m <<= s;                                   // leading bit 62 (s >= 0)
  m += s <= 30 ? (long long)__float2int_rn(f * __int_as_float((127 + s) << 23))
               : __float2ll_rn(f * __int_as_float((127 + s) << 23));
  if (m < (1ull << 62)) {
    m <<= 1;
    s++;
  }
  m = (m + 511 + ((m >> 10) & 1)) >> 10;     // 53 bits, to nearest, ties to even
  const int E = 1085 + sexp - s;             // value = m 2^(sexp - s + 10), 2^52 <= m <= 2^53
  if (E < 1 || E > 2045) {
    const double r = scale_slow((double)m, sexp - s + 10);
    return a < 0 ? -r : r;
  }
  return __longlong_as_double((long long)(((unsigned long long)(E - 1) << 52) + m | (unsigned long long)a & 1ull << 63));
}

__device__ __forceinline__ double flip(double x) {
  return __longlong_as_double(__double_as_longlong(x) ^ (long long)(1ull << 63));
}

__global__ void __launch_bounds__(NT, 1)
oz_kernel(const __grid_constant__ OzMaps maps, OzShape g, const int* __restrict__ eL, const int* __restrict__ eN,
          double* __restrict__ out, int* err) {
  extern __shared__ __align__(1024) unsigned char smem_raw[];
  unsigned char* smem = (unsigned char*)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
  uint64_t* bars = (uint64_t*)(smem + STAGES * STAGE);
  uint32_t* tmem_slot = (uint32_t*)(bars + 17);
  const uint32_t sbase = smem_u32(smem), bar0 = smem_u32(bars);
  auto FULL = [&](int s) { return bar0 + 8u * s; };
  auto EMPTY = [&](int s) { return bar0 + 8u * (2 + s); };
  // accumulator c (C_0 .. C_4, and 5: C_5 + C_6 + C_7): complete, drained
  auto AFULL = [&](int c) { return bar0 + 8u * (4 + c); };
  auto AEMPTY = [&](int c) { return bar0 + 8u * (10 + c); };
  const uint32_t DONE = bar0 + 8u * 16;

  __shared__ int abort_flag;
  if (threadIdx.x == 0) abort_flag = *(volatile int*)err;
  __syncthreads();
  if (abort_flag) return;   // an earlier CTA gave up a wait: skip the work
  const int warp = __shfl_sync(0xffffffffu, (int)threadIdx.x >> 5, 0), lane = threadIdx.x & 31;
  if (threadIdx.x == 0) {
    for (int s = 0; s < 2; s++) {
      mbar_init(FULL(s), 1);
      mbar_init(EMPTY(s), 1);
    }
    for (int c = 0; c < NACC; c++) {
      mbar_init(AFULL(c), 1);
      mbar_init(AEMPTY(c), EPI_W);
    }
    mbar_init(DONE, 1);
    mbar_fence_init();
  }
  if (warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_slot)),
                 "r"(512)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = __shfl_sync(0xffffffffu, *tmem_slot, 0);
  const int nchunk = (g.nst + CHUNK_ST - 1) / CHUNK_ST;
  // unit -> (batch entry, lane tile, column tile), column tiles fastest: CTAs side by side share the lane tile
  auto decode = [&](long u, int& b, int& li, int& ni) {
    const unsigned r = (unsigned)u / (unsigned)g.tn;
    ni = (int)((unsigned)u - r * (unsigned)g.tn);
    b = (int)(r / (unsigned)g.tl);
    li = (int)(r - (unsigned)b * (unsigned)g.tl);
  };

  // (warps 0 and 1 keep all lanes in their loops and elect one per batch of
  // copies or MMAs: see tc_gemm.cu)
  if (warp == 0) {
    {
      uint32_t it = 0;
      bool ok = true;
      for (long u = blockIdx.x; u < g.units && ok; u += gridDim.x) {
        int b, li, ni;
        decode(u, b, li, ni);
        for (int st = 0; st < g.nst; st++, it++) {
          const uint32_t sl = it & 1;
          if (!mbar_wait_uniform(EMPTY(sl), ((it >> 1) & 1) ^ 1, err, 2)) { ok = false; break; }
          if (elect_one()) {
            mbar_expect_tx(FULL(sl), STAGE);
            tma_load_3d(sbase + sl * STAGE, &maps.l, FULL(sl), st * TK, li * TL, b * ND);
            tma_load_3d(sbase + sl * STAGE + ND * LPL, &maps.n, FULL(sl), st * TK, ni * TN, b * ND);
          }
          __syncwarp();
        }
      }
      // the copies still in flight land before the CTA exits (on the normal path they have)
      const uint32_t n = it < 2 ? it : 2;
      for (uint32_t j = it - n; j < it; j++) mbar_drain(FULL(j & 1), (j >> 1) & 1);
    }
  } else if (warp == 1) {
    {
      const uint64_t d0 = desc64(sbase);
      constexpr uint64_t PL = LPL >> 4, PC = CPL >> 4;
      uint32_t it = 0, ch = 0;
      bool ok = true;
      for (long u = blockIdx.x; u < g.units && ok; u += gridDim.x) {
        for (int c = 0; c < nchunk && ok; c++, ch++) {
          const int st1 = min(g.nst, (c + 1) * CHUNK_ST);
          for (int st = c * CHUNK_ST; st < st1; st++, it++) {
            const uint32_t sl = it & 1;
            const bool first = st == c * CHUNK_ST, last = st == st1 - 1;
            if (!mbar_wait_uniform(FULL(sl), (it >> 1) & 1, err, 8)) { ok = false; break; }
            tc_fence_after();
            const uint64_t al = d0 + ((sl * STAGE) >> 4), bn = al + ((ND * LPL) >> 4);
#pragma unroll
            for (int c6 = 0; c6 < NACC; c6++) {
              if (first) {
                if (!mbar_wait_uniform(AEMPTY(c6), (ch & 1) ^ 1, err, 4)) { ok = false; break; }
                tc_fence_after();
              }
              if (elect_one()) {
#pragma unroll
                for (int cl = c6 == 5 ? 7 : c6; cl >= c6; cl--)      // C_7, C_6, C_5
#pragma unroll
                  for (int s = cl == 7; s <= min(cl, ND - 1); s++)
#pragma unroll
                    for (int kk = 0; kk < 2; kk++)
                      mma_bf16(tmem + c6 * TN, al + s * PL + 2 * kk, bn + (cl - s) * PC + 2 * kk,
                               !(first && (cl < 5 || cl == 7) && s == (cl == 7) && kk == 0));
                if (last) commit(AFULL(c6));
                if (c6 == NACC - 1) commit(EMPTY(sl));
              }
              __syncwarp();
            }
            if (!ok) break;
          }
        }
      }
      // every MMA issued complete before TMEM is released
      if (elect_one()) commit(DONE);
      __syncwarp();
      mbar_drain(DONE, 0);
    }
  } else if (warp >= EPI0) {
    const int q = warp & 3, h = (warp - EPI0) >> 2;         // lane quadrant, column quarter
    const uint32_t tl = tmem + ((uint32_t)(32 * q) << 16) + EC * h;
    uint32_t ch = 0;
    bool ok = true;
    for (long u = blockIdx.x; u < g.units && ok; u += gridDim.x) {
      int b, li, ni;
      decode(u, b, li, ni);
      long long acc[EC];
      float rest[EC];
#pragma unroll
      for (int j = 0; j < EC; j++) {
        acc[j] = 0;
        rest[j] = 0.f;
      }
      for (int c = 0; c < nchunk; c++, ch++) {
        // class c holds integers in units of 2^(-9 c); in units of C_3 they count 2^(27 - 9 c)
#pragma unroll
        for (int c6 = 0; c6 < NACC; c6++) {
          // (every lane polls: the sleeping wait of one lane woke up to 250 ns late, six times a chunk)
          if (!__all_sync(0xffffffffu, mbar_wait(AFULL(c6), ch & 1, err, 16))) { ok = false; break; }
          tc_fence_after();
#pragma unroll
          for (int f = 0; f < EC; f += EH) {
            float v[EH];
            tmem_ld10(tl + c6 * TN + f, v);
            if (f + EH == EC) {
              tc_fence_before();
              __syncwarp();
              if (lane == 0) mbar_arrive(AEMPTY(c6));
            }
#pragma unroll
            for (int j = 0; j < EH; j++) {
              if (c6 < 4) {
                acc[f + j] += (long long)__float2int_rn(v[j] * (float)(1 << (9 * (c6 & 3)))) * (1 << (27 - 9 * (c6 & 3)));
              } else if (c6 == 4) {
                const float x4 = v[j] * 0x1p27f;   // C_4 in units of C_3, a multiple of 2^-9
                const int n4 = __float2int_rn(x4);
                acc[f + j] += n4;
                rest[f + j] += x4 - (float)n4;
              } else {
                rest[f + j] = fmaf(v[j], 0x1p27f, rest[f + j]);
              }
            }
          }
        }
        if (!ok) break;
      }
      if (!ok) break;
      const int i = li * TL + 32 * q + lane, j0 = ni * TN + EC * h;
      if (i < g.nl) {
        const int ei = eL[(long)b * g.el + (i >> g.lsh)];
        // biased exponents E: 2^(E - 1022) above the row; value = 2^(e_l + e_n - 16 - 27) (acc + rest)
        const int es = ei - 2 * 1022 - 43;
        const int* en = eN + (long)b * g.en;
#pragma unroll
        for (int j = 0; j < EC; j += 2) {
          const int col = j0 + j;
          if (col < g.nn) {
            const bool two = col + 1 < g.nn;
            const int e0 = en[col >> g.nsh], e1 = two ? en[(col + 1) >> g.nsh] : 0;
            double x = round_sum(acc[j], rest[j], es + e0), y = two ? round_sum(acc[j + 1], rest[j + 1], es + e1) : 0.0;
            if (ei == NB_ROW || e0 == NB_ROW) x = __longlong_as_double(0x7ff8000000000000ll);
            if (ei == NB_ROW || e1 == NB_ROW) y = __longlong_as_double(0x7ff8000000000000ll);
            if (g.alpha < 0) {
              x = flip(x);
              y = flip(y);
            }
            if (g.pairs) {
              reinterpret_cast<double2*>(out)[(long)b * g.sbo + (long)(col >> 1) * g.ldo + i] = make_double2(x, y);
            } else {
              double* o = out + (long)b * g.sbo + (long)col * g.ldo + i;
              if (g.acc) {
                o[0] += x;
                if (two) o[g.ldo] += y;
              } else {
                o[0] = x;
                if (two) o[g.ldo] = y;
              }
            }
          }
        }
      }
      __syncwarp();
    }
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  if (warp == 1)
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(512) : "memory");
}

// ---------------------------------------------------------------------------
// operand preparation
// ---------------------------------------------------------------------------

__device__ __forceinline__ int expo(double x) { return (__double2hiint(x) >> 20) & 0x7ff; }

// Largest biased exponent of each row: element (r, k) at src[r lr + k lk], CX
// doubles each.  Rows with contiguous K: one warp per row.
template <int CX>
__global__ void __launch_bounds__(256) oz_exp_rows(const double* __restrict__ src, long sb, long lr, int rows, int K,
                                                   int* __restrict__ e) {
  const int r = blockIdx.x * 8 + (threadIdx.x >> 5), lane = threadIdx.x & 31;
  if (r >= rows) return;
  const double* p = src + ((long)blockIdx.y * sb + (long)r * lr) * CX;
  int m = 0;
  for (int k = lane; k < K * CX; k += 32) m = max(m, expo(p[k]));
  for (int o = 16; o > 0; o >>= 1) m = max(m, __shfl_xor_sync(0xffffffffu, m, o));
  if (lane == 0) e[(long)blockIdx.y * rows + r] = m;
}

// The same for contiguous rows (stride lk along K): one thread per row, K in
// slices of KS rows over blockIdx.y, merged by atomicMax (e zeroed before).
constexpr int KS = 64;
template <int CX>
__global__ void __launch_bounds__(128) oz_exp_cols(const double* __restrict__ src, long sb, long lk, int rows, int K,
                                                   int* __restrict__ e) {
  const int r = blockIdx.x * 128 + threadIdx.x;
  if (r >= rows) return;
  const int k0 = blockIdx.y * KS, k1 = min(K, k0 + KS);
  const double* p = src + ((long)blockIdx.z * sb + (long)k0 * lk + r) * CX;
  int m = 0;
#pragma unroll 4
  for (int k = k0; k < k1; k++, p += lk * CX) {
    if (CX == 2) {
      const double2 v = *reinterpret_cast<const double2*>(p);
      m = max(m, max(expo(v.x), expo(v.y)));
    } else {
      m = max(m, expo(p[0]));
    }
  }
  atomicMax(e + (long)blockIdx.z * rows + r, m);
}

// x 2^(62 - e), rounded, for a row of biased exponent E (e = E - 1022): |result| <= 2^62.
__device__ __forceinline__ long long fixed62(double x, int E) {
  const unsigned long long u = (unsigned long long)__double_as_longlong(x);
  const int ex = (int)(u >> 52) & 0x7ff;
  unsigned long long m = (u & 0xfffffffffffffull) | (ex ? 1ull << 52 : 0);
  const int sh = max(ex, 1) - E + 9;
  if (sh >= 0) m <<= min(sh, 10);
  else m = sh > -55 ? (m + (1ull << (-sh - 1))) >> -sh : 0;
  return (long long)u < 0 ? -(long long)m : (long long)m;
}

// The planes of 8 consecutive reals of a row: digits from the last, each
// balanced digit taken off with its carry; the plane value 2^(-9 s) d is formed
// by adding d to the bits of 1.5 2^(23 - 9 s) and subtracting that number.
// EMB: x holds 4 complex values, and the two rows (re, -im) and (im, re) are written.
template <bool EMB>
__device__ __forceinline__ void put8(const double* x, int E, uint16_t* dst, long plane, int ldp) {
  long long f[8];
#pragma unroll
  for (int i = 0; i < 8; i++) f[i] = E == NB_ROW ? 0 : fixed62(x[i], E);
#pragma unroll
  for (int s = ND - 1; s >= 0; s--) {
    uint32_t v[8];
#pragma unroll
    for (int i = 0; i < 8; i++) {
      int d;
      if (s > 0) {
        f[i] += 256;
        d = ((int)f[i] & 511) - 256;
        f[i] >>= 9;
      } else {
        d = (int)f[i];
      }
      const float big = __int_as_float(0x4B400000 - ((9 * s) << 23));   // 1.5 2^(23 - 9 s)
      v[i] = __float_as_uint(__fsub_rn(__int_as_float(__float_as_int(big) + d), big));
    }
    uint32_t w[4];
#pragma unroll
    for (int i = 0; i < 4; i++) w[i] = __byte_perm(v[2 * i], v[2 * i + 1], 0x7632);
    uint16_t* o = dst + s * plane;
    if (EMB) {
      *reinterpret_cast<uint4*>(o) =
          make_uint4(w[0] ^ 0x80000000u, w[1] ^ 0x80000000u, w[2] ^ 0x80000000u, w[3] ^ 0x80000000u);
#pragma unroll
      for (int i = 0; i < 4; i++) w[i] = __byte_perm(w[i], 0, 0x1032);
      *reinterpret_cast<uint4*>(o + ldp) = make_uint4(w[0], w[1], w[2], w[3]);
    } else {
      *reinterpret_cast<uint4*>(o) = make_uint4(w[0], w[1], w[2], w[3]);
    }
  }
}

// Digit planes dst[b][s][row][ldp] of an operand (K-contiguous rows): one
// thread per 8 reals.  conj negates imaginary parts.
template <int CX, bool EMB>
__global__ void __launch_bounds__(256) oz_slice_rows(const double* __restrict__ src, long sb, long lr, int rows, int K,
                                                     int conj, const int* __restrict__ e, uint16_t* __restrict__ dst,
                                                     int ldp) {
  const int ng = (K * CX + 7) / 8;
  const long i = (long)blockIdx.x * 256 + threadIdx.x;
  if (i >= (long)rows * ng) return;
  const int r = (int)(i / ng), k0 = (int)(i % ng) * (8 / CX);
  const long b = blockIdx.y;
  const double* p = src + (b * sb + (long)r * lr + k0) * CX;
  double x[8];
#pragma unroll
  for (int j = 0; j < 8 / CX; j++) {
    const bool in = k0 + j < K;
    if (CX == 2) {
      const double2 v = in ? *reinterpret_cast<const double2*>(p + 2 * j) : make_double2(0.0, 0.0);
      x[2 * j] = v.x;
      x[2 * j + 1] = conj ? flip(v.y) : v.y;
    } else {
      x[j] = in ? p[j] : 0.0;
    }
  }
  const long plane = (long)rows * (EMB ? 2 : 1) * ldp;
  put8<EMB>(x, e[b * rows + r], dst + b * ND * plane + (long)r * (EMB ? 2 : 1) * ldp + k0 * CX, plane, ldp);
}

// The same for row-contiguous sources (stride lk along K): a block turns a
// tile of 32 rows by 8 / CX x 8 K values around in shared memory.
template <int CX, bool EMB>
__global__ void __launch_bounds__(256) oz_slice_cols(const double* __restrict__ src, long sb, long lk, int rows, int K,
                                                     int conj, const int* __restrict__ e, uint16_t* __restrict__ dst,
                                                     int ldp) {
  constexpr int KT = 64 / CX;                       // 64 reals of K
  __shared__ double t[KT][33 * CX];
  const int r0 = blockIdx.x * 32, k0 = blockIdx.y * KT;
  const long b = blockIdx.z;
  for (int i = threadIdx.x; i < KT * 32; i += 256) {
    const int k = i / 32, r = i % 32;
    const bool in = k0 + k < K && r0 + r < rows;
    const double* p = src + (b * sb + (long)(k0 + k) * lk + r0 + r) * CX;
    if (CX == 2) {
      const double2 v = in ? *reinterpret_cast<const double2*>(p) : make_double2(0.0, 0.0);
      t[k][2 * r] = v.x;
      t[k][2 * r + 1] = conj ? flip(v.y) : v.y;
    } else {
      t[k][r] = in ? p[0] : 0.0;
    }
  }
  __syncthreads();
  const int r = threadIdx.x / 8, c = threadIdx.x % 8;  // 8 reals of K each
  if (r0 + r >= rows || k0 * CX + 8 * c >= ldp) return;
  double x[8];
#pragma unroll
  for (int j = 0; j < 8 / CX; j++) {
    if (CX == 2) {
      x[2 * j] = t[4 * c + j][2 * r];
      x[2 * j + 1] = t[4 * c + j][2 * r + 1];
    } else {
      x[j] = t[8 * c + j][r];
    }
  }
  const long plane = (long)rows * (EMB ? 2 : 1) * ldp;
  put8<EMB>(x, e[b * rows + r0 + r], dst + b * ND * plane + (long)(r0 + r) * (EMB ? 2 : 1) * ldp + k0 * CX + 8 * c,
            plane, ldp);
}

// One operand of a product: `rows` rows of K elements, element (r, k) at
// src[r lr + k lk] (one of lr, lk is 1), batch entries sb elements apart.
struct Side {
  const double* src;
  int rows;
  long lr, lk, sb;
  bool conj, emb;
};

int pad8i(int x) { return (x + 7) & ~7; }

long plane_rows(const Side& s) { return s.emb ? 2L * s.rows : s.rows; }

template <int CX>
cudaError_t prepare(const Side& a, int K, int batch, int* e, uint16_t* pl, cudaStream_t s) {
  const int ldp = pad8i(K * CX);
  if (a.lk == 1) {
    oz_exp_rows<CX><<<dim3((a.rows + 7) / 8, batch), 256, 0, s>>>(a.src, a.sb, a.lr, a.rows, K, e);
    const unsigned nb = (unsigned)(((long)a.rows * (ldp / 8) + 255) / 256);
    if (a.emb)
      oz_slice_rows<2, true><<<dim3(nb, batch), 256, 0, s>>>(a.src, a.sb, a.lr, a.rows, K, a.conj, e, pl, ldp);
    else
      oz_slice_rows<CX, false><<<dim3(nb, batch), 256, 0, s>>>(a.src, a.sb, a.lr, a.rows, K, a.conj, e, pl, ldp);
  } else {
    cudaError_t st = cudaMemsetAsync(e, 0, sizeof(int) * (size_t)batch * a.rows, s);
    if (st != cudaSuccess) return st;
    oz_exp_cols<CX><<<dim3((a.rows + 127) / 128, (K + KS - 1) / KS, batch), 128, 0, s>>>(a.src, a.sb, a.lk, a.rows, K,
                                                                                        e);
    const dim3 grid((a.rows + 31) / 32, (K * CX + 63) / 64, batch);
    if (a.emb)
      oz_slice_cols<2, true><<<grid, 256, 0, s>>>(a.src, a.sb, a.lk, a.rows, K, a.conj, e, pl, ldp);
    else
      oz_slice_cols<CX, false><<<grid, 256, 0, s>>>(a.src, a.sb, a.lk, a.rows, K, a.conj, e, pl, ldp);
  }
  return cudaGetLastError();
}

// [batch x 7 planes][rows][ldp] bf16 read as boxes of 7 planes x `box` rows x 32 K.
cudaError_t plane_map(CUtensorMap* map, const void* base, int batch, long rows, int Kr, int ldp, int box) {
  static const PFN_cuTensorMapEncodeTiled_v12000 enc = [] {
    void* p = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault, &q) != cudaSuccess ||
        q != cudaDriverEntryPointSuccess)
      p = nullptr;
    return (PFN_cuTensorMapEncodeTiled_v12000)p;
  }();
  if (!enc) return cudaErrorNotSupported;
  cuuint64_t dims[3] = {(cuuint64_t)Kr, (cuuint64_t)rows, (cuuint64_t)batch * ND};
  cuuint64_t strides[2] = {(cuuint64_t)ldp * 2, (cuuint64_t)ldp * 2 * rows};
  cuuint32_t bx[3] = {TK, (cuuint32_t)box, ND};
  cuuint32_t estr[3] = {1, 1, 1};
  return enc(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 3, (void*)base, dims, strides, bx, estr,
             CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_64B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
             CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS
             ? cudaSuccess
             : cudaErrorInvalidValue;
}

size_t align256(size_t x) { return (x + 255) & ~(size_t)255; }

// Scratch of one operand: exponents, then planes.
size_t side_bytes(long rows, long prow, int Kr, int batch) {
  return align256(sizeof(int) * (size_t)rows * batch) + align256(2 * (size_t)ND * prow * pad8i(Kr) * batch);
}

template <int CX>
cudaError_t launch(const OzMaps& maps, const OzShape& g, const int* eL, const int* eN, double* out, const OzWork& w,
                   cudaStream_t s) {
  int dev = 0, nsm = 0;
  if (g.units >= (1L << 31)) return cudaErrorInvalidValue;   // counted in 32 bits
  cudaError_t e = cudaGetDevice(&dev);
  if (e == cudaSuccess) e = cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev);
  if (e == cudaSuccess) e = cudaFuncSetAttribute(oz_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)SMEM);
  if (e != cudaSuccess) return e;
  oz_kernel<<<(unsigned)std::min<long>(g.units, nsm), NT, SMEM, s>>>(maps, g, eL, eN, out, w.err());
  if (w.launches) ++*w.launches;
  return cudaGetLastError();
}

// One slab: lane planes pL with exponents eL against column planes pN, eN.
template <int CX>
cudaError_t slab(const Side& l, const Side& n, int K, int nb, const int* eL, const uint16_t* pL, const int* eN,
                 const uint16_t* pN, double* out, long ldo, long sbo, bool pairs, double alpha, bool acc, const OzWork& w,
                 cudaStream_t s) {
  const int Kr = K * CX, ldp = pad8i(Kr);
  OzMaps maps;
  cudaError_t e = plane_map(&maps.n, pN, nb, plane_rows(n), Kr, ldp, TN);
  if (e == cudaSuccess) e = plane_map(&maps.l, pL, nb, plane_rows(l), Kr, ldp, TL);
  if (e != cudaSuccess) return e;
  OzShape g;
  g.nl = (int)plane_rows(l);
  g.nn = (int)plane_rows(n);
  g.nst = (Kr + TK - 1) / TK;
  g.tl = (g.nl + TL - 1) / TL;
  g.tn = (g.nn + TN - 1) / TN;
  g.lsh = l.emb;
  g.nsh = n.emb;
  g.el = l.rows;
  g.en = n.rows;
  g.units = (long)nb * g.tl * g.tn;
  g.pairs = pairs;
  g.acc = acc;
  g.alpha = alpha;
  g.ldo = ldo;
  g.sbo = sbo;
  return launch<CX>(maps, g, eL, eN, out, w, s);
}

// Whether a complex product embeds A (as the columns) or B (as the lanes).
// The time of the two choices, in units of 1 / 152 of a tile's 114 cycles per
// real K: the tiles, and the planes of both operands (22 bytes read and
// written per real at 6.5 TB/s).
bool embed_a(int M, int N) {
  auto cost = [](long lanes, long cols) {
    return (double)((lanes + TL - 1) / TL) * ((cols + TN - 1) / TN) + 0.009 * (lanes + cols);
  };
  return cost(N, 2L * M) <= cost(2L * N, M);
}

thread_local long long g_limit = -1;   // test hook: most scratch of a product

// Scratch for planes and exponents.
size_t room_of(const OzWork& w) {
  const size_t b = g_limit < 0 ? w.bytes : std::min(w.bytes, (size_t)g_limit);
  return b > HEAD ? b - HEAD : 0;
}

// Slabs of a product that fit in `room` bytes: batch entries, lane rows and
// column rows of each (of the sides' own rows).
struct Slabs {
  int bs, lrows, nrows;
};

// Whole batch entries where one fits, as even as they go; else whole tiles of
// one entry: column tiles in up to half the room, lane tiles in what is left.
// Rows are rounded down to tiles, so that room for one tile of each side is
// enough and more of it never fails.
bool plan_slabs(int lrows, bool lemb, int nrows, bool nemb, int Kr, int batch, size_t room, Slabs& p) {
  auto lane = [&](int nb, int r) { return side_bytes(r, lemb ? 2L * r : r, Kr, nb); };
  auto col = [&](int nb, int r) { return side_bytes(r, nemb ? 2L * r : r, Kr, nb); };
  // the largest n <= most for which fits(n), 0 where there is none
  auto largest = [](int most, auto fits) {
    int lo = 0, hi = most + 1;
    while (lo + 1 < hi) {
      const int mid = lo + (hi - lo) / 2;
      if (fits(mid)) lo = mid;
      else hi = mid;
    }
    return lo;
  };
  p = Slabs{1, lrows, nrows};
  const int bs = largest(batch, [&](int nb) { return lane(nb, lrows) + col(nb, nrows) <= room; });
  if (bs > 0) {
    const int parts = (batch + bs - 1) / bs;
    p.bs = (batch + parts - 1) / parts;
    return true;
  }
  const int lt = TL >> lemb, nt = TN >> nemb;   // rows of a tile
  const size_t lane1 = lane(1, std::min(lt, lrows));
  if (lane1 + col(1, std::min(nt, nrows)) > room) return false;
  const int ct = std::max(1, largest((nrows + nt - 1) / nt, [&](int t) {
    const size_t c = col(1, (int)std::min<long>(nrows, (long)t * nt));
    return c <= room / 2 && c + lane1 <= room;
  }));
  p.nrows = (int)std::min<long>(nrows, (long)ct * nt);
  const size_t left = room - col(1, p.nrows);
  const int rt = largest((lrows + lt - 1) / lt,
                         [&](int t) { return lane(1, (int)std::min<long>(lrows, (long)t * lt)) <= left; });
  p.lrows = (int)std::min<long>(lrows, (long)rt * lt);
  return true;
}

// out(lane i, column j) over batch entries, in slabs that fit the scratch.
// pairs: the N side is embedded and out is complex [j / 2][i].
template <int CX>
cudaError_t product(Side L, Side N, int K, int batch, double* out, long ldo, long sbo, bool pairs, double alpha,
                    bool acc, const OzWork& w, cudaStream_t s) {
  if (L.rows <= 0 || N.rows <= 0 || batch <= 0) return cudaSuccess;
  if (K <= 0 || (long)K * CX > OZ_MAX_K) return cudaErrorInvalidValue;   // the int64 sums stay below 2^62
  const int Kr = K * CX;
  Slabs pl;
  if (!plan_slabs(L.rows, L.emb, N.rows, N.emb, Kr, batch, room_of(w), pl))
    return cudaErrorMemoryAllocation;
  const int bs = pl.bs, lrows = pl.lrows, nrows = pl.nrows;
  for (int b0 = 0; b0 < batch; b0 += bs) {
    const int nb = std::min(bs, batch - b0);
    for (int n0 = 0; n0 < N.rows; n0 += nrows) {
      Side n = N;
      n.src += ((long)b0 * N.sb + (long)n0 * N.lr) * CX;
      n.rows = std::min(nrows, N.rows - n0);
      int* eN = (int*)(w.buf + HEAD);
      uint16_t* pN = (uint16_t*)((unsigned char*)eN + align256(sizeof(int) * (size_t)n.rows * nb));
      cudaError_t e = prepare<CX>(n, K, nb, eN, pN, s);
      if (e != cudaSuccess) return e;
      if (w.launches) *w.launches += 2;
      unsigned char* lbuf = (unsigned char*)eN + side_bytes(n.rows, plane_rows(n), Kr, nb);
      for (int l0 = 0; l0 < L.rows; l0 += lrows) {
        Side l = L;
        l.src += ((long)b0 * L.sb + (long)l0 * L.lr) * CX;
        l.rows = std::min(lrows, L.rows - l0);
        int* eL = (int*)lbuf;
        uint16_t* pL = (uint16_t*)(lbuf + align256(sizeof(int) * (size_t)l.rows * nb));
        if ((e = prepare<CX>(l, K, nb, eL, pL, s)) != cudaSuccess) return e;
        if (w.launches) *w.launches += 2;
        // pairs: double2 units along rows; embedded lanes: two doubles per complex column
        double* o = out + (pairs ? 2 * ((long)b0 * sbo + (long)n0 * ldo + l0)
                                 : (long)b0 * sbo + (long)n0 * ldo + (L.emb ? 2L : 1L) * l0);
        if ((e = slab<CX>(l, n, K, nb, eL, pL, eN, pN, o, ldo, sbo, pairs, alpha, acc, w, s)) != cudaSuccess) return e;
      }
    }
  }
  return cudaSuccess;
}

}  // namespace

size_t oz_work_bytes(int M, int N, int K, int batch) {
  const long small = std::min(M, N), big = std::max(M, N);
  return HEAD + side_bytes(small, 2 * small, 2 * K, batch) + side_bytes(big, big, 2 * K, batch);
}

size_t oz_work_min(int K) { return HEAD + side_bytes(TN, TN, 2 * K, 1) + side_bytes(TL, TL, 2 * K, 1); }

bool oz_fits(int M, int N, int K, int batch, bool real, const OzWork& w) {
  const bool ea = !real && embed_a(M, N);
  const int Kr = real ? K : 2 * K;
  Slabs p;
  return w.buf && Kr <= OZ_MAX_K && plan_slabs(N, !real && !ea, M, ea, Kr, batch, room_of(w), p);
}

void oz_limit(long long bytes) { g_limit = bytes; }

bool oz_plan(int M, int N, int K, int batch, bool real, size_t bytes, int plan[3]) {
  const bool ea = !real && embed_a(M, N);
  Slabs p;
  const bool ok = plan_slabs(N, !real && !ea, M, ea, real ? K : 2 * K, batch, bytes > HEAD ? bytes - HEAD : 0, p);
  plan[0] = p.bs;
  plan[1] = p.nrows;
  plan[2] = p.lrows;
  return ok;
}

cudaError_t oz_alloc(OzWork& w, size_t want, size_t least, cudaStream_t s) {
  cudaError_t e = cudaErrorMemoryAllocation;
  for (w.bytes = std::max(want, least);; w.bytes = std::max(least, w.bytes / 2)) {
    e = cudaMalloc((void**)&w.buf, w.bytes);
    if (e != cudaErrorMemoryAllocation) break;
    cudaGetLastError();
    w.buf = nullptr;
    if (w.bytes <= least) break;
  }
  if (e == cudaSuccess) e = cudaMemsetAsync(w.buf, 0, 64, s);
  if (e != cudaSuccess) oz_free(w);
  return e;
}

void oz_free(OzWork& w) {
  if (w.buf) cudaFree(w.buf);
  w = OzWork{};
}

// The FP64 kernel takes 4.3 us per unit of K and round of its 64 x 64 tiles
// over the SMs (two multiply-adds a clock on each): 35 us for one tile of
// K = 8, and 0.3 ms for one of K = 71.  The digit form's five launches are
// about 35 us in all.
bool oz_wins(int M, int N, int K, int batch) {
  const double tiles = ((M + 63) / 64) * (double)((N + 63) / 64) * batch;
  return ceil(tiles / 152.0) * K >= 10.0 && 2L * K <= OZ_MAX_K;
}

cudaError_t oz_gemm_z(int la, int lb, int M, int N, int K, const double2* A, int lda, long sA, const double2* B,
                      int ldb, long sB, double2* C, int ldc, long sC, int batch, const OzWork& w, cudaStream_t s) {
  Side a{(const double*)A, M, la == A_KM ? 1L : (long)lda, la == A_KM ? (long)lda : 1L, sA, la == A_MK_CONJ, false};
  Side b{(const double*)B, N, lb == B_KN ? 1L : (long)ldb, lb == B_KN ? (long)ldb : 1L, sB, lb == B_NK_CONJ, false};
  if (embed_a(M, N)) {
    // embedded A as the columns, lanes along N: out[m][n] one double2 per lane
    a.emb = true;
    return product<2>(b, a, K, batch, (double*)C, ldc, sC, true, 1.0, false, w, s);
  }
  // embedded B as the lanes (real columns of the interleaved C), plain A rows as the columns
  b.emb = true;
  return product<2>(b, a, K, batch, (double*)C, 2L * ldc, 2 * sC, false, 1.0, false, w, s);
}

cudaError_t gemm_z_best(int la, int lb, int M, int N, int K, const double2* A, int lda, long sA, const double2* B,
                        int ldb, long sB, double2* C, int ldc, long sC, int batch, const OzWork& w, cudaStream_t s) {
  if (oz_wins(M, N, K, batch) && oz_fits(M, N, K, batch, false, w))
    return oz_gemm_z(la, lb, M, N, K, A, lda, sA, B, ldb, sB, C, ldc, sC, batch, w, s);
  if (w.launches) ++*w.launches;
  return gemm_z(la, lb, M, N, K, A, lda, sA, B, ldb, sB, C, ldc, sC, batch, s);
}

bool oz_lanes_fit(int M, int K, const OzWork& w) { return w.buf && side_bytes(M, 2L * M, 2 * K, 1) <= room_of(w); }

size_t oz_lane_bytes(int N, int K) { return side_bytes(N, N, 2 * K, 1); }

cudaError_t oz_lane_prepare(const double2* B, int ldb, int N, int K, void* lanes, cudaStream_t s) {
  if (2L * K > OZ_MAX_K) return cudaErrorInvalidValue;
  const Side b{(const double*)B, N, 1L, (long)ldb, 0, false, false};
  return prepare<2>(b, K, 1, (int*)lanes, (uint16_t*)((unsigned char*)lanes + align256(sizeof(int) * (size_t)N)), s);
}

cudaError_t oz_gemm_z_lanes(int la, int M, int N, int K, const double2* A, int lda, const void* lanes, double2* C,
                            int ldc, const OzWork& w, cudaStream_t s) {
  if (!oz_lanes_fit(M, K, w)) return cudaErrorMemoryAllocation;
  const Side a{(const double*)A, M, la == A_KM ? 1L : (long)lda, la == A_KM ? (long)lda : 1L, 0, la == A_MK_CONJ, true};
  const Side b{nullptr, N, 1L, 1L, 0, false, false};
  int* eA = (int*)(w.buf + HEAD);
  uint16_t* pA = (uint16_t*)((unsigned char*)eA + align256(sizeof(int) * (size_t)M));
  const cudaError_t e = prepare<2>(a, K, 1, eA, pA, s);
  if (e != cudaSuccess) return e;
  return slab<2>(b, a, K, 1, (const int*)lanes,
                 (const uint16_t*)((const unsigned char*)lanes + align256(sizeof(int) * (size_t)N)), eA, pA, (double*)C,
                 ldc, 0, true, 1.0, false, w, s);
}

cudaError_t oz_gemm_d(bool a_km, bool b_kn, int M, int N, int K, const double* A, long lda, const double* B, long ldb,
                      double* C, long ldc, double alpha, bool acc, const OzWork& w, cudaStream_t s) {
  Side a{A, M, a_km ? 1L : lda, a_km ? lda : 1L, 0, false, false};
  Side b{B, N, b_kn ? 1L : ldb, b_kn ? ldb : 1L, 0, false, false};
  return product<1>(b, a, K, 1, C, ldc, 0, false, alpha, acc, w, s);
}
