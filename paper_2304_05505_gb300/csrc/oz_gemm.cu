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
// That is an error relative to the largest entries of the two rows.  Where a
// row's large entries all meet small ones of the other row, as those of a
// compact basis function far from an orbital, sum |a||b| is far below their
// product and an FP64 loop would do better.  So every product is checked
// first: with m = |x| 2^-e of every entry (bf16, of the larger of re and im),
// S = sum m_a m_b per result, in one product on the tensor cores.  The digits'
// roundings, 2^-62 / sqrt(12) rms each, add up to 2^-63.3 (|m_a|^2 + |m_b|^2)^(1/2)
// of the product of the largest entries at most.  So where S is below
// 2^-10 (|m_a|^2 + |m_b|^2)^(1/2), seven digits are not enough.  Measured rms errors
// in u sum |a||b| (u = 2^-53), K = 100 to 6000: dense rows 0.05 to 0.01 where the
// FP64 pipe's sums leave 0.5; one large entry beside small ones, S at 2^-8 of the
// root, 0.4 to 0.7 where they leave 4 to 6.  (A line that knows S alone would not
// do: at S = 2^-10 rows with one large entry each leave 0.5, but rows of 1200
// small ones beside it 10.)
// Tiles with more than a few such results go to a second form of the kernel:
// eight digits (71 bits), classes up to C_8, good down to a line of 2^-18.  What
// is below that, what few there are in a tile, and results whose rows hold a NaN
// or an Inf are computed in FP64: single entries by a warp each, tiles with a
// majority of them as gemm_z computes them.  Below the first line lie 0.05 to
// 0.15 % of S4b's results for Gaussians of 0.25 to 3.5 bohr^-2, but 20 % for the
// benzene cells' basis, 10 % of S1's and S4a's and 58 % of THC-AO-K's; below the
// second 0.07 % at most.  (The same in FP64 instead of eight digits: THC-AO-K of
// the benzene cell at 4 x 4 x 4 k 401 ms, 31 now; its build 25.8 and 11.1 ms, and 9.5
// for the wider Gaussians, which took 8.8 unchecked.)
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
// The form with eight digits: 43 digit products, tiles of 128 x 64, whose eight
// accumulators (C_0 .. C_6, and C_7 + C_8) fill TMEM, an int64 and an int per output;
// 1.45 times the time of the other per output.
// The integer epilogue keeps the FP64 pipe (2 results per SM and clock) out of
// the kernel: conversion and rounding of an output are about 30 integer
// instructions.
#include "oz_gemm.cuh"
#include "mbarrier.cuh"

#include <cuda.h>
#include <cudaTypedefs.h>

#include <algorithm>

namespace {

constexpr int TL = 128, TN = 80, TK = 32;              // lane rows, column rows, K of a stage
constexpr uint32_t LPL = TL * TK * 2;                  // bytes of a lane plane tile: 8 KB
constexpr int STAGES = 2;
constexpr int CHUNK_ST = 2;                            // stages of an exact chunk (64 K)
constexpr int EPI0 = 4, EPI_W = 16, NT = 32 * (EPI0 + EPI_W);
// The two forms: 7 digits, and 8 for tiles that the check gives to them.
template <bool W>
struct Form {
  static constexpr int ND = W ? 8 : 7;                 // digits
  static constexpr int CMAX = W ? 8 : 7;               // the last class
  static constexpr int N = W ? 64 : TN;                // columns of a tile
  static constexpr int NACC = W ? 8 : 6;               // accumulators: the last classes share one
  static constexpr uint32_t CPL = N * TK * 2;          // bytes of a column plane tile
  static constexpr uint32_t STAGE = ND * (LPL + CPL);  // 91 KB, 96 KB
  static constexpr size_t SMEM = STAGES * STAGE + 1024 + 256;
  static constexpr int EC = N / 4, EH = EC / 2;        // columns of an epilogue warp, and of a read of them
  static_assert(SMEM <= 232448 && NACC * N <= 512, "227 KB of shared memory per block, 512 TMEM columns");
};
constexpr int WN = Form<true>::N;
constexpr int NB_ROW = 2047;                           // biased exponent of a row with a NaN or an Inf
constexpr size_t HEAD = 256;                           // bytes before scratch of its own: the error block

// The check of a product: stages of 64 K of the magnitudes, 128B swizzle
constexpr int MK = 64;
constexpr uint32_t MLB = TL * MK * 2, MCB = TN * MK * 2, MSTAGE = MLB + MCB;   // 16 KB + 10 KB
constexpr int MSTAGES = 6, MEPI = 8, MNT = 32 * (4 + MEPI);
constexpr size_t MSMEM = MSTAGES * MSTAGE + 1024 + 256;
constexpr float CHECK7 = 0x1p20f, CHECK8 = 0x1p36f;    // digits are not enough where S^2 CHECK < |m_a|^2 + |m_b|^2
constexpr int FEW = 16;                                // entries of a warp's 32 x 40 up to which 7 digits and FP64 do
constexpr int MANY = 800;                              // and from which the tile goes whole in FP64
constexpr int EPU = 512;                               // room for single entries, per tile
constexpr float NORM_UNIT = 4096.f;                    // |m|^2 is counted in units of 2^-12

struct OzMaps {
  CUtensorMap l, n;
};

// What the check leaves: cnt[0] tiles (flag bit 0, listed in tiles) and cnt[1]
// entries (tile, lane row << 8 | column row of it) to be computed in FP64, and
// cnt[2] tiles (flag bit 1) to be computed with 8 digits.
struct OzList {
  int *cnt, *flag, *tiles;
  uint2* ents;
  int cap;
};

struct OzShape {
  int lr, nr;        // rows of the two sides, and of a tile (an embedded row counts two)
  int lt, nt;
  int mst;           // stages of the check
  int nl, nn;        // valid lanes (rows of the lane operand) and columns
  int nst;           // K stages
  int tl, tn;        // tiles
  int ftn;           // column tiles of the flags
  int nd;            // digit planes in memory
  int lsh, nsh;      // exponent index = row >> sh (embedded operands: pairs of rows share one)
  long el, en;       // exponents per batch entry
  long units;
  int pairs;         // columns 2m, 2m + 1 are the real and imaginary part of output row m
  int acc;           // add to out
  double alpha;
  long ldo, sbo;     // doubles (pairs: double2)
};

// unit -> (batch entry, lane tile, column tile), column tiles fastest: CTAs side by side share the lane tile
__device__ __forceinline__ void decode(const OzShape& g, long u, int& b, int& li, int& ni) {
  const unsigned r = (unsigned)u / (unsigned)g.tn;
  ni = (int)((unsigned)u - r * (unsigned)g.tn);
  b = (int)(r / (unsigned)g.tl);
  li = (int)(r - (unsigned)b * (unsigned)g.tl);
}

template <int N>
__device__ __forceinline__ void mma_bf16(uint32_t d, uint64_t a, uint64_t b, uint32_t accumulate) {
  // kind::f16, D f32 (bit 4), A and B bf16 (bits 7 and 10), K-major, N >> 3 at bit 17, M >> 4 at bit 24
  constexpr uint32_t idesc =
      (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(N >> 3) << 17) | ((uint32_t)(TL >> 4) << 24);
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

// 8 or 10 consecutive columns of this thread's TMEM lane (half of an epilogue warp's: registers).
__device__ __forceinline__ void tmem_ld8(uint32_t t, float* v) {
  uint32_t r[8];
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];\n"
      "tcgen05.wait::ld.sync.aligned;"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7])
      : "r"(t)
      : "memory");
#pragma unroll
  for (int i = 0; i < 8; i++) v[i] = __uint_as_float(r[i]);
}
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

template <bool W>
__global__ void __launch_bounds__(NT, 1)
oz_kernel(const __grid_constant__ OzMaps maps, OzShape g, const int* __restrict__ eL, const int* __restrict__ eN,
          double* __restrict__ out, OzList f, int* err) {
  typedef Form<W> F;
  constexpr int ND = F::ND, NACC = F::NACC, EC = F::EC, EH = F::EH, N = F::N;
  constexpr uint32_t STAGE = F::STAGE, CPL = F::CPL;
  if (W && f.cnt[2] == 0) return;
  extern __shared__ __align__(1024) unsigned char smem_raw[];
  unsigned char* smem = (unsigned char*)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
  uint64_t* bars = (uint64_t*)(smem + STAGES * STAGE);
  uint32_t* tmem_slot = (uint32_t*)(bars + 5 + 2 * NACC);
  const uint32_t sbase = smem_u32(smem), bar0 = smem_u32(bars);
  auto FULL = [&](int s) { return bar0 + 8u * s; };
  auto EMPTY = [&](int s) { return bar0 + 8u * (2 + s); };
  // accumulator c (one class each, the last C_5 + C_6 + C_7 or C_7 + C_8): complete, drained
  auto AFULL = [&](int c) { return bar0 + 8u * (4 + c); };
  auto AEMPTY = [&](int c) { return bar0 + 8u * (4 + NACC + c); };
  const uint32_t DONE = bar0 + 8u * (4 + 2 * NACC);

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
  // tiles that the check has left to FP64 or to the other form are passed over by every warp
  const bool holes = W || (f.cnt && (f.cnt[0] | f.cnt[2]) != 0);
  auto pass = [&](long u) {
    if (!holes) return false;
    if (!W) return f.flag[u] != 0;
    int b, li, ni;
    decode(g, u, b, li, ni);
    const int* fl = f.flag + ((long)b * g.tl + li) * g.ftn;
    const int n0 = ni * N / TN, n1 = min((ni * N + N - 1) / TN, g.ftn - 1);
    return ((fl[n0] | fl[n1]) & 2) == 0;
  };
  static_assert(N <= TN, "a tile of the wide form meets at most two of the flags'");

  // (warps 0 and 1 keep all lanes in their loops and elect one per batch of
  // copies or MMAs: see tc_gemm.cu)
  if (warp == 0) {
    {
      uint32_t it = 0;
      bool ok = true;
      for (long u = blockIdx.x; u < g.units && ok; u += gridDim.x) {
        if (pass(u)) continue;
        int b, li, ni;
        decode(g, u, b, li, ni);
        for (int st = 0; st < g.nst; st++, it++) {
          const uint32_t sl = it & 1;
          if (!mbar_wait_uniform(EMPTY(sl), ((it >> 1) & 1) ^ 1, err, 2)) { ok = false; break; }
          if (elect_one()) {
            mbar_expect_tx(FULL(sl), STAGE);
            tma_load_3d(sbase + sl * STAGE, &maps.l, FULL(sl), st * TK, li * TL, b * g.nd);
            tma_load_3d(sbase + sl * STAGE + ND * LPL, &maps.n, FULL(sl), st * TK, ni * N, b * g.nd);
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
        if (pass(u)) continue;
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
                constexpr auto top = [](int c) { return c == NACC - 1 ? F::CMAX : c; };
                constexpr auto s0 = [](int cl) { return cl < ND ? 0 : cl - ND + 1; };
#pragma unroll
                for (int cl = top(c6); cl >= c6; cl--)               // the smaller classes first
#pragma unroll
                  for (int s = s0(cl); s <= min(cl, ND - 1); s++)
#pragma unroll
                    for (int kk = 0; kk < 2; kk++)
                      mma_bf16<N>(tmem + c6 * N, al + s * PL + 2 * kk, bn + (cl - s) * PC + 2 * kk,
                                  !(first && cl == top(c6) && s == s0(cl) && kk == 0));
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
      if (pass(u)) continue;
      int b, li, ni;
      decode(g, u, b, li, ni);
      long long acc[EC];
      float rest[EC];
      int lo[W ? EC : 1];
#pragma unroll
      for (int j = 0; j < EC; j++) {
        acc[j] = 0;
        rest[j] = 0.f;
        if (W) lo[W ? j : 0] = 0;
      }
      for (int c = 0; c < nchunk; c++, ch++) {
        // class c holds integers in units of 2^(-9 c); in units of C_3 they count 2^(27 - 9 c).
        // 8 digits: lo holds what is below C_3 in units of C_6, 0 <= lo < 2^27, and rest what is below that
#pragma unroll
        for (int c6 = 0; c6 < NACC; c6++) {
          // (every lane polls: the sleeping wait of one lane woke up to 250 ns late, six times a chunk)
          if (!__all_sync(0xffffffffu, mbar_wait(AFULL(c6), ch & 1, err, 16))) { ok = false; break; }
          tc_fence_after();
#pragma unroll
          for (int f = 0; f < EC; f += EH) {
            float v[EH];
            if constexpr (EH == 8) tmem_ld8(tl + c6 * N + f, v);
            else tmem_ld10(tl + c6 * N + f, v);
            if (f + EH == EC) {
              tc_fence_before();
              __syncwarp();
              if (lane == 0) mbar_arrive(AEMPTY(c6));
            }
#pragma unroll
            for (int j = 0; j < EH; j++) {
              if (c6 < 4) {
                acc[f + j] += (long long)__float2int_rn(v[j] * (float)(1 << (9 * (c6 & 3)))) * (1 << (27 - 9 * (c6 & 3)));
              } else if (W) {
                int& l = lo[W ? f + j : 0];
                if (c6 < 7) {
                  const int n = __float2int_rn(v[j] * (c6 == 4 ? 0x1p36f : c6 == 5 ? 0x1p45f : 0x1p54f));
                  if (c6 == 4) {
                    acc[f + j] += n >> 9;
                    l += (n & 511) << 18;
                  } else if (c6 == 5) {
                    acc[f + j] += n >> 18;
                    l += (n & 0x3ffff) << 9;
                  } else {
                    l += n;
                  }
                } else {
                  const float x = fmaf(v[j], 0x1p54f, rest[f + j]);
                  const int n = __float2int_rn(x);
                  rest[f + j] = x - (float)n;
                  l += n;
                  acc[f + j] += l >> 27;
                  l &= (1 << 27) - 1;
                }
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
      const int i = li * TL + 32 * q + lane, j0 = ni * N + EC * h;
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
            auto value = [&](int j, int sexp) {
              if constexpr (W) {
                // in units of C_6 while that fits 62 bits
                if (acc[j] < (1ll << 34) && acc[j] >= -(1ll << 34))
                  return round_sum(acc[j] * (1 << 27) + lo[j], rest[j], sexp - 27);
                return round_sum(acc[j], (float)lo[j] * 0x1p-27f, sexp);
              } else {
                return round_sum(acc[j], rest[j], sexp);
              }
            };
            double x = value(j, es + e0), y = two ? value(j + 1, es + e1) : 0.0;
            if (!f.cnt) {   // (else rows with a NaN or an Inf are left to FP64)
              if (ei == NB_ROW || e0 == NB_ROW) x = __longlong_as_double(0x7ff8000000000000ll);
              if (ei == NB_ROW || e1 == NB_ROW) y = __longlong_as_double(0x7ff8000000000000ll);
            }
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
// the check, and what it leaves to FP64
// ---------------------------------------------------------------------------

// K-major tile of 64 bf16, 128B swizzle, 8-row groups 1024 B apart.
__device__ __forceinline__ uint64_t desc128(uint32_t addr) {
  return (uint64_t)((addr & 0x3FFFF) >> 4) | ((uint64_t)1 << 16) | ((uint64_t)(1024 >> 4) << 32) | ((uint64_t)1 << 46) |
         ((uint64_t)2 << 61);
}

// S of every entry, tiles as in oz_kernel<false> (rows of an embedded side counted
// once, so its box is half used): warp 0 loads, warp 1 multiplies into one of
// two accumulators, warps 4-11 compare (32 lanes x 40 columns each).  It reads
// a fifteenth of the product's planes and multiplies a 68th to a 136th as much.
__global__ void __launch_bounds__(MNT, 1)
oz_check_kernel(const __grid_constant__ OzMaps maps, OzShape g, const int* __restrict__ eL, const int* __restrict__ eN,
                const unsigned* __restrict__ qL, const unsigned* __restrict__ qN, OzList f, int* err) {
  extern __shared__ __align__(1024) unsigned char smem_raw[];
  unsigned char* smem = (unsigned char*)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
  uint64_t* bars = (uint64_t*)(smem + MSTAGES * MSTAGE);
  uint32_t* tmem_slot = (uint32_t*)(bars + 17);
  const uint32_t sbase = smem_u32(smem), bar0 = smem_u32(bars);
  auto FULL = [&](int s) { return bar0 + 8u * s; };
  auto EMPTY = [&](int s) { return bar0 + 8u * (6 + s); };
  auto AFULL = [&](int c) { return bar0 + 8u * (12 + c); };
  auto AEMPTY = [&](int c) { return bar0 + 8u * (14 + c); };
  const uint32_t DONE = bar0 + 8u * 16;
  static_assert(MSTAGES == 6, "barrier slots");

  __shared__ int abort_flag;
  if (threadIdx.x == 0) abort_flag = *(volatile int*)err;
  __syncthreads();
  if (abort_flag) return;
  const int warp = __shfl_sync(0xffffffffu, (int)threadIdx.x >> 5, 0), lane = threadIdx.x & 31;
  if (threadIdx.x == 0) {
    for (int s = 0; s < MSTAGES; s++) {
      mbar_init(FULL(s), 1);
      mbar_init(EMPTY(s), 1);
    }
    for (int c = 0; c < 2; c++) {
      mbar_init(AFULL(c), 1);
      mbar_init(AEMPTY(c), MEPI);
    }
    mbar_init(DONE, 1);
    mbar_fence_init();
  }
  if (warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_slot)),
                 "r"(256)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = __shfl_sync(0xffffffffu, *tmem_slot, 0);

  if (warp == 0) {
    uint32_t it = 0;
    bool ok = true;
    for (long u = blockIdx.x; u < g.units && ok; u += gridDim.x) {
      int b, li, ni;
      decode(g, u, b, li, ni);
      for (int st = 0; st < g.mst; st++, it++) {
        const uint32_t sl = it % MSTAGES;
        if (!mbar_wait_uniform(EMPTY(sl), ((it / MSTAGES) & 1) ^ 1, err, 2)) { ok = false; break; }
        if (elect_one()) {
          mbar_expect_tx(FULL(sl), MSTAGE);
          tma_load_3d(sbase + sl * MSTAGE, &maps.l, FULL(sl), st * MK, li * g.lt, b);
          tma_load_3d(sbase + sl * MSTAGE + MLB, &maps.n, FULL(sl), st * MK, ni * g.nt, b);
        }
        __syncwarp();
      }
    }
    // the copies still in flight land before the CTA exits
    const uint32_t n = it < MSTAGES ? it : MSTAGES;
    for (uint32_t j = it - n; j < it; j++) mbar_drain(FULL(j % MSTAGES), (j / MSTAGES) & 1);
  } else if (warp == 1) {
    uint32_t it = 0, local = 0;
    bool ok = true;
    for (long u = blockIdx.x; u < g.units && ok; u += gridDim.x, local++) {
      const uint32_t set = local & 1;
      if (!mbar_wait_uniform(AEMPTY(set), ((local >> 1) & 1) ^ 1, err, 4)) break;
      for (int st = 0; st < g.mst; st++, it++) {
        const uint32_t sl = it % MSTAGES;
        if (!mbar_wait_uniform(FULL(sl), (it / MSTAGES) & 1, err, 8)) { ok = false; break; }
        tc_fence_after();
        const uint64_t al = desc128(sbase + sl * MSTAGE), bn = desc128(sbase + sl * MSTAGE + MLB);
        if (elect_one()) {
#pragma unroll
          for (int kk = 0; kk < MK / 16; kk++) mma_bf16<TN>(tmem + 128 * set, al + 2 * kk, bn + 2 * kk, st > 0 || kk > 0);
          commit(EMPTY(sl));
          if (st == g.mst - 1) commit(AFULL(set));
        }
        __syncwarp();
      }
    }
    // every MMA issued complete before TMEM is released
    if (elect_one()) commit(DONE);
    __syncwarp();
    mbar_drain(DONE, 0);
  } else if (warp >= 4) {
    const int q = warp & 3, h = (warp - 4) >> 2;            // lane quadrant, column half
    constexpr int MC = TN / 2;
    const uint32_t tl = tmem + ((uint32_t)(32 * q) << 16) + MC * h;
    uint32_t local = 0;
    for (long u = blockIdx.x; u < g.units; u += gridDim.x, local++) {
      int b, li, ni;
      decode(g, u, b, li, ni);
      const uint32_t set = local & 1;
      // rows with a NaN or an Inf: of this lane, and of the columns as bits
      const int r = 32 * q + lane, c0 = MC * h;
      const bool row = r < g.lt && li * g.lt + r < g.lr;
      const bool nb = row && eL[(long)b * g.el + li * g.lt + r] == NB_ROW;
      const float ql = row ? (float)qL[(long)b * g.el + li * g.lt + r] : 0.f;
      auto column = [&](int c) { return c < g.nt && ni * g.nt + c < g.nr; };
      auto norm = [&](int c) { return column(c) ? (float)qN[(long)b * g.en + ni * g.nt + c] : 0.f; };
      const float qn0 = norm(c0 + lane), qn1 = lane < MC - 32 ? norm(c0 + 32 + lane) : 0.f;
      auto bad = [&](int c) { return column(c) && eN[(long)b * g.en + ni * g.nt + c] == NB_ROW; };
      const unsigned long long cols = (unsigned long long)__ballot_sync(0xffffffffu, column(c0 + lane)) |
                                      (unsigned long long)__ballot_sync(0xffffffffu, lane < MC - 32 && column(c0 + 32 + lane)) << 32;
      unsigned long long m = (unsigned long long)__ballot_sync(0xffffffffu, bad(c0 + lane)) |
                             (unsigned long long)__ballot_sync(0xffffffffu, lane < MC - 32 && bad(c0 + 32 + lane)) << 32;
      if (nb) m = ~0ull;
      unsigned long long m7 = m;               // what 7 digits are not enough for; m: nor 8
      if (!__all_sync(0xffffffffu, mbar_wait(AFULL(set), (local >> 1) & 1, err, 16))) break;
      tc_fence_after();
#pragma unroll
      for (int j0 = 0; j0 < MC; j0 += 10) {
        float v[10];
        tmem_ld10(tl + 128 * set + j0, v);
#pragma unroll
        for (int j = 0; j < 10; j++) {
          const float q = ql + __shfl_sync(0xffffffffu, j0 + j < 32 ? qn0 : qn1, (j0 + j) & 31);   // (by every lane)
          const float w = v[j] * v[j] * NORM_UNIT;
          if (v[j] > 0.f && w * CHECK7 < q) m7 |= 1ull << (j0 + j);
          if (v[j] > 0.f && w * CHECK8 < q) m |= 1ull << (j0 + j);
        }
      }
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(AEMPTY(set));
      m7 = row ? m7 & cols : 0ull;
      const int all7 = (int)__reduce_add_sync(0xffffffffu, (unsigned)__popcll(m7));
      if (all7 == 0) continue;
      m &= m7;
      const bool wide = all7 > FEW;          // the tile with 8 digits, entries beyond those in FP64
      if (!wide) m = m7;
      const int mine = __popcll(m), all = (int)__reduce_add_sync(0xffffffffu, (unsigned)mine);
      bool whole = g.acc || all > MANY;      // (an entry that is added to cannot be overwritten later)
      if (!whole && all > 0) {
        int off = mine;
        for (int o = 1; o < 32; o <<= 1) {
          const int t = __shfl_up_sync(0xffffffffu, off, o);
          if (lane >= o) off += t;
        }
        int base = 0;
        if (lane == 0) base = atomicAdd(f.cnt + 1, all);
        base = __shfl_sync(0xffffffffu, base, 0);
        whole = base < 0 || base > f.cap - all;   // no room: the slots up to cap are left empty
        for (int i = base + off - mine; m && base >= 0; m &= m - 1, i++)
          if (i < f.cap)
            f.ents[i] = whole ? make_uint2(~0u, 0u)
                              : make_uint2((unsigned)u, (unsigned)(r << 8 | (c0 + __ffsll((long long)m) - 1)));
      }
      if (lane == 0) {
        const int bits = (whole ? 1 : 0) | (wide ? 2 : 0), old = bits ? atomicOr(f.flag + u, bits) : 0;
        if (bits & ~old & 1) f.tiles[atomicAdd(f.cnt, 1)] = (int)u;
        if (bits & ~old & 2) atomicAdd(f.cnt + 2, 1);
      }
    }
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  if (warp == 1)
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(256) : "memory");
}

// A side in memory: element (r, k) of batch entry b at src[b sb + r lr + k lk].
struct Source {
  const double* src;
  long sb, lr, lk;
  bool conj;
};

template <int CX>
struct Num;
template <>
struct Num<1> {
  double x;
  __device__ __forceinline__ void fma_(const Num& a, const Num& b) { x = fma(a.x, b.x, x); }
  __device__ __forceinline__ void add(int o) { x += __shfl_xor_sync(0xffffffffu, x, o); }
};
template <>
struct Num<2> {
  double x, y;
  // the order of gemm_z
  __device__ __forceinline__ void fma_(const Num& a, const Num& b) {
    x = fma(a.x, b.x, x);
    x = fma(-a.y, b.y, x);
    y = fma(a.x, b.y, y);
    y = fma(a.y, b.x, y);
  }
  __device__ __forceinline__ void add(int o) {
    x += __shfl_xor_sync(0xffffffffu, x, o);
    y += __shfl_xor_sync(0xffffffffu, y, o);
  }
};

template <int CX>
__device__ __forceinline__ Num<CX> element(const Source& s, int b, int r, int k) {
  const double* p = s.src + (b * s.sb + r * s.lr + k * s.lk) * CX;
  if constexpr (CX == 2) {
    const double2 v = *reinterpret_cast<const double2*>(p);
    return Num<2>{v.x, s.conj ? -v.y : v.y};
  } else {
    return Num<1>{*p};
  }
}

template <int CX>
__device__ __forceinline__ void put(double* __restrict__ out, const OzShape& g, int b, int r, int c, Num<CX> v) {
  const double sg = g.alpha < 0 ? -1.0 : 1.0;
  if constexpr (CX == 2) {
    // embedded columns: double2 along the rows; embedded lanes: two doubles a row
    double* o = out + (g.pairs ? 2 * (b * g.sbo + c * g.ldo + r) : b * g.sbo + c * g.ldo + 2L * r);
    *reinterpret_cast<double2*>(o) = make_double2(sg * v.x, sg * v.y);
  } else {
    double* o = out + b * g.sbo + c * g.ldo + r;
    *o = g.acc ? *o + sg * v.x : sg * v.x;
  }
}

// The listed tiles (32 LI rows x 8 CJ columns, a block each, as gemm_kernel
// sums them) and entries (a warp each).  Two FP64 multiply-adds a clock and SM
// bind both, so entries are listed one by one up to 800 of a warp's 1280 (from
// 80 on as tiles: up to 16 times the work, on the SMs that get the tiles).
template <int CX, int LI, int CJ>
__global__ void __launch_bounds__(256) oz_exact_kernel(Source l, Source n, int K, OzShape g, OzList f,
                                                       double* __restrict__ out, const int* err) {
  typedef Num<CX> T;
  constexpr int BK = 8, R = 32 * LI, C = 8 * CJ;
  __shared__ T ls[BK][R + 1], ns[BK][C + 1];
  const int ntile = f.cnt[0], nent = (int)min((unsigned)f.cnt[1], (unsigned)f.cap);
  if ((ntile | nent) == 0 || *(volatile const int*)err) return;
  const int tx = threadIdx.x & 31, ty = threadIdx.x >> 5;
  for (int t = blockIdx.x; t < ntile; t += gridDim.x) {
    int b, li, ni;
    decode(g, f.tiles[t], b, li, ni);
    const int r0 = li * R, c0 = ni * C;
    T acc[LI][CJ];
#pragma unroll
    for (int i = 0; i < LI; i++)
#pragma unroll
      for (int j = 0; j < CJ; j++) acc[i][j] = T{};
    for (int k0 = 0; k0 < K; k0 += BK) {
      for (int e = threadIdx.x; e < R * BK; e += 256) {
        const int kk = l.lk == 1 ? e % BK : e / R, r = l.lk == 1 ? e / BK : e % R;
        ls[kk][r] = r0 + r < g.lr && k0 + kk < K ? element<CX>(l, b, r0 + r, k0 + kk) : T{};
      }
      for (int e = threadIdx.x; e < C * BK; e += 256) {
        const int kk = n.lk == 1 ? e % BK : e / C, c = n.lk == 1 ? e / BK : e % C;
        ns[kk][c] = c0 + c < g.nr && k0 + kk < K ? element<CX>(n, b, c0 + c, k0 + kk) : T{};
      }
      __syncthreads();
#pragma unroll
      for (int kk = 0; kk < BK; kk++) {
        T lv[LI];
#pragma unroll
        for (int i = 0; i < LI; i++) lv[i] = ls[kk][tx + 32 * i];
#pragma unroll
        for (int j = 0; j < CJ; j++) {
          const T nv = ns[kk][ty + 8 * j];
#pragma unroll
          for (int i = 0; i < LI; i++) acc[i][j].fma_(nv, lv[i]);
        }
      }
      __syncthreads();
    }
#pragma unroll
    for (int i = 0; i < LI; i++)
#pragma unroll
      for (int j = 0; j < CJ; j++) {
        const int r = r0 + tx + 32 * i, c = c0 + ty + 8 * j;
        if (r < g.lr && c < g.nr) put<CX>(out, g, b, r, c, acc[i][j]);
      }
  }
  for (int i = blockIdx.x * 8 + ty; i < nent; i += gridDim.x * 8) {
    const uint2 e = f.ents[i];
    if (e.x == ~0u || (f.flag[e.x] & 1)) continue;
    int b, li, ni;
    decode(g, e.x, b, li, ni);
    const int r = li * R + (int)(e.y >> 8), c = ni * C + (int)(e.y & 255);
    T v{};
#pragma unroll 4
    for (int k = tx; k < K; k += 32) v.fma_(element<CX>(n, b, c, k), element<CX>(l, b, r, k));
    for (int o = 16; o > 0; o >>= 1) v.add(o);
    if (tx == 0) put<CX>(out, g, b, r, c, v);
  }
}

// ---------------------------------------------------------------------------
// operand preparation
// ---------------------------------------------------------------------------

__device__ __forceinline__ int expo(double x) { return (__double2hiint(x) >> 20) & 0x7ff; }

// Largest biased exponent of each row: element (r, k) at src[r lr + k lk], CX
// doubles each.  Rows with contiguous K: one warp per row.  (The sums of the
// magnitudes' squares, sq, are set to zero for the slicing that follows.)
template <int CX>
__global__ void __launch_bounds__(256) oz_exp_rows(const double* __restrict__ src, long sb, long lr, int rows, int K,
                                                   int* __restrict__ e, unsigned* __restrict__ sq) {
  const int r = blockIdx.x * 8 + (threadIdx.x >> 5), lane = threadIdx.x & 31;
  if (r >= rows) return;
  const double* p = src + ((long)blockIdx.y * sb + (long)r * lr) * CX;
  int m = 0;
  for (int k = lane; k < K * CX; k += 32) m = max(m, expo(p[k]));
  for (int o = 16; o > 0; o >>= 1) m = max(m, __shfl_xor_sync(0xffffffffu, m, o));
  if (lane == 0) {
    e[(long)blockIdx.y * rows + r] = m;
    sq[(long)blockIdx.y * rows + r] = 0u;
  }
}

// The same for contiguous rows (stride lk along K): one thread per row, K in
// slices of KS rows over blockIdx.y, merged by atomicMax (e and sq zeroed before).
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

// x 2^(71 - e), rounded, for a row of biased exponent E (e = E - 1022), as hi 2^27 + lo, 0 <= lo < 2^27.
__device__ __forceinline__ void fixed71(double x, int E, long long& hi, int& lo) {
  const unsigned long long u = (unsigned long long)__double_as_longlong(x);
  const int ex = (int)(u >> 52) & 0x7ff;
  unsigned long long m = (u & 0xfffffffffffffull) | (ex ? 1ull << 52 : 0);
  const int sh = max(ex, 1) - E + 18;                // at most 19
  if (sh >= 0) {
    lo = (int)(m << min(sh, 19)) & 0x7ffffff;
    hi = (long long)(m >> (27 - min(sh, 19)));
  } else {
    m = sh > -55 ? (m + (1ull << (-sh - 1))) >> -sh : 0;
    lo = (int)m & 0x7ffffff;
    hi = (long long)(m >> 27);
  }
  if ((long long)u < 0) {
    hi = -hi - (lo != 0);
    lo = -lo & 0x7ffffff;
  }
}

// x 2^(62 - e), rounded.
__device__ __forceinline__ long long fixed62(double x, int E) {
  const unsigned long long u = (unsigned long long)__double_as_longlong(x);
  const int ex = (int)(u >> 52) & 0x7ff;
  unsigned long long m = (u & 0xfffffffffffffull) | (ex ? 1ull << 52 : 0);
  const int sh = max(ex, 1) - E + 9;
  if (sh >= 0) m <<= min(sh, 10);
  else m = sh > -55 ? (m + (1ull << (-sh - 1))) >> -sh : 0;
  return (long long)u < 0 ? -(long long)m : (long long)m;
}

// u 2^-e (u: the bits of a nonnegative double of a row of biased exponent E) truncated to bf16; at least 2^-41 for u > 0.
__device__ __forceinline__ uint32_t mag16(unsigned long long u, int E) {
  const int ex = (int)(u >> 52), d = E - ex;
  if (u == 0 || E == NB_ROW) return 0;
  return ex == 0 || d > 40 ? 86u << 7 : (uint32_t)(126 - d) << 7 | (uint32_t)(u >> 45 & 0x7f);
}

// The magnitudes of 8 consecutive reals of a row (CX = 2: of 4 complex values); the sum of their squares.
template <int CX>
__device__ __forceinline__ unsigned put_mags(const double* x, int E, uint16_t* dst) {
  uint32_t w[4 / CX];
  float q = 0.f;
#pragma unroll
  for (int i = 0; i < 4 / CX; i++) {
    uint32_t v[2];
#pragma unroll
    for (int j = 0; j < 2; j++) {
      const double* y = x + (2 * i + j) * CX;
      unsigned long long u = (unsigned long long)__double_as_longlong(y[0]) & ~(1ull << 63);
      if (CX == 2) u = max(u, (unsigned long long)__double_as_longlong(y[CX - 1]) & ~(1ull << 63));
      v[j] = mag16(u, E);
      const float m = __uint_as_float(v[j] << 16);
      q = fmaf(m, m, q);
    }
    w[i] = v[0] | v[1] << 16;
  }
  if constexpr (CX == 2) *reinterpret_cast<uint2*>(dst) = make_uint2(w[0], w[1]);
  else *reinterpret_cast<uint4*>(dst) = make_uint4(w[0], w[1], w[2], w[3]);
  return __float2uint_rn(q * NORM_UNIT);
}

// The planes of 8 consecutive reals of a row: digits from the last, each
// balanced digit taken off with its carry; the plane value 2^(-9 s) d is formed
// by adding d to the bits of 1.5 2^(23 - 9 s) and subtracting that number.
// ND: 7, or 8 digits (whose first seven are the value rounded to 62 bits: balanced digits).
// EMB: x holds 4 complex values, and the two rows (re, -im) and (im, re) are written.
template <bool EMB, int ND>
__device__ __forceinline__ void put8(const double* x, int E, uint16_t* dst, long plane, int ldp) {
  long long f[8];
  int l[8];
#pragma unroll
  for (int i = 0; i < 8; i++) {
    f[i] = 0;
    l[i] = 0;
    if (E != NB_ROW) {
      if constexpr (ND == 8) fixed71(x[i], E, f[i], l[i]);
      else f[i] = fixed62(x[i], E);
    }
  }
#pragma unroll
  for (int s = ND - 1; s >= 0; s--) {
    uint32_t v[8];
#pragma unroll
    for (int i = 0; i < 8; i++) {
      int d;
      if (ND == 8 && s > 4) {
        l[i] += 256;
        d = (l[i] & 511) - 256;
        l[i] >>= 9;
        if (s == 5) f[i] += l[i];
      } else if (s > 0) {
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
// thread per 8 reals.  conj negates imaginary parts.  ND = 8: also the magnitudes.
template <int CX, bool EMB, int ND>
__global__ void __launch_bounds__(256) oz_slice_rows(const double* __restrict__ src, long sb, long lr, int rows, int K,
                                                     int conj, const int* __restrict__ e, uint16_t* __restrict__ dst,
                                                     int ldp, uint16_t* __restrict__ mag, int ldm,
                                                     unsigned* __restrict__ sq) {
  const int ng = (K * CX + 7) / 8;
  const long i = (long)blockIdx.x * 256 + threadIdx.x;
  const unsigned act = __ballot_sync(0xffffffffu, i < (long)rows * ng);
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
  const int E = e[b * rows + r];
  put8<EMB, ND>(x, E, dst + b * ND * plane + (long)r * (EMB ? 2 : 1) * ldp + k0 * CX, plane, ldp);
  if (ND == 8) {
    // (integer sums: the same whatever their order)
    const unsigned q = put_mags<CX>(x, E, mag + (b * rows + r) * ldm + k0);
    int one;
    __match_all_sync(act, r, &one);
    if (one) {                     // (the same for every lane: a row of its own)
      const unsigned w = __reduce_add_sync(act, q);
      if ((threadIdx.x & 31) == 0) atomicAdd(sq + b * rows + r, w);   // (lane 0 is the first to have work)
    } else {
      atomicAdd(sq + b * rows + r, q);
    }
  }
}

// The same for row-contiguous sources (stride lk along K): a block turns a
// tile of 32 rows by 8 / CX x 8 K values around in shared memory.
template <int CX, bool EMB, int ND>
__global__ void __launch_bounds__(256) oz_slice_cols(const double* __restrict__ src, long sb, long lk, int rows, int K,
                                                     int conj, const int* __restrict__ e, uint16_t* __restrict__ dst,
                                                     int ldp, uint16_t* __restrict__ mag, int ldm,
                                                     unsigned* __restrict__ sq) {
  constexpr int KT = 64 / CX;                       // 64 reals of K
  __shared__ double t[KT][33 * CX];
  __shared__ unsigned part[32];
  if (threadIdx.x < 32) part[threadIdx.x] = 0u;
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
  const bool in = r0 + r < rows && k0 * CX + 8 * c < ldp;
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
  if (in) {
    const int E = e[b * rows + r0 + r];
    put8<EMB, ND>(x, E, dst + b * ND * plane + (long)(r0 + r) * (EMB ? 2 : 1) * ldp + k0 * CX + 8 * c, plane, ldp);
    if (ND == 8) atomicAdd(part + r, put_mags<CX>(x, E, mag + (b * rows + r0 + r) * ldm + k0 + 8 / CX * c));
  }
  if (ND == 7) return;
  __syncthreads();
  if (threadIdx.x < 32 && r0 + (int)threadIdx.x < rows) atomicAdd(sq + b * rows + r0 + threadIdx.x, part[threadIdx.x]);
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

size_t align256(size_t x) { return (x + 255) & ~(size_t)255; }

// Scratch of one operand: exponents, sums of the magnitudes' squares, digit
// planes, magnitudes (null: none are made).
struct Planes {
  int* e;
  unsigned* sq;
  uint16_t *pl, *mag;
};

size_t exp_bytes(long rows, int batch) { return align256(2 * sizeof(int) * (size_t)rows * batch); }
size_t digit_bytes(long rows, bool emb, int K, int CX, int batch, int nd = 8) {
  return align256(2 * (size_t)nd * (rows << emb) * pad8i(K * CX) * batch);
}
size_t side_bytes(long rows, bool emb, int K, int CX, int batch) {
  return exp_bytes(rows, batch) + digit_bytes(rows, emb, K, CX, batch) + align256(2 * (size_t)rows * pad8i(K) * batch);
}

Planes planes_at(void* at, long rows, bool emb, int K, int CX, int batch) {
  unsigned char* p = (unsigned char*)at + exp_bytes(rows, batch);
  return Planes{(int*)at, (unsigned*)at + rows * batch, (uint16_t*)p, (uint16_t*)(p + digit_bytes(rows, emb, K, CX, batch))};
}

long tiles_of(long rows, bool emb, int t) { return ((rows << emb) + t - 1) / t; }

// Scratch of the check's list, for `units` tiles.
size_t list_bytes(long units) { return align256(64 + 2 * sizeof(int) * (size_t)units) + align256(sizeof(uint2) * EPU * (size_t)units); }

OzList list_at(void* at, long units) {
  OzList f;
  f.cnt = (int*)at;
  f.flag = f.cnt + 16;
  f.tiles = f.flag + units;
  f.ents = (uint2*)((unsigned char*)at + align256(64 + 2 * sizeof(int) * (size_t)units));
  f.cap = (int)std::min<long>(EPU * units, 0x7fffff00L);
  return f;
}

template <int CX, int ND>
cudaError_t prepare_digits(const Side& a, int K, int batch, const Planes& p, cudaStream_t s) {
  const int ldp = pad8i(K * CX), ldm = pad8i(K);
  if (a.lk == 1) {
    oz_exp_rows<CX><<<dim3((a.rows + 7) / 8, batch), 256, 0, s>>>(a.src, a.sb, a.lr, a.rows, K, p.e, p.sq);
    const unsigned nb = (unsigned)(((long)a.rows * (ldp / 8) + 255) / 256);
    if (a.emb)
      oz_slice_rows<2, true, ND><<<dim3(nb, batch), 256, 0, s>>>(a.src, a.sb, a.lr, a.rows, K, a.conj, p.e, p.pl, ldp, p.mag,
                                                             ldm, p.sq);
    else
      oz_slice_rows<CX, false, ND><<<dim3(nb, batch), 256, 0, s>>>(a.src, a.sb, a.lr, a.rows, K, a.conj, p.e, p.pl, ldp,
                                                               p.mag, ldm, p.sq);
  } else {
    cudaError_t st = cudaMemsetAsync(p.e, 0, 2 * sizeof(int) * (size_t)batch * a.rows, s);   // p.sq too
    if (st != cudaSuccess) return st;
    oz_exp_cols<CX><<<dim3((a.rows + 127) / 128, (K + KS - 1) / KS, batch), 128, 0, s>>>(a.src, a.sb, a.lk, a.rows, K,
                                                                                        p.e);
    const dim3 grid((a.rows + 31) / 32, (K * CX + 63) / 64, batch);
    if (a.emb)
      oz_slice_cols<2, true, ND><<<grid, 256, 0, s>>>(a.src, a.sb, a.lk, a.rows, K, a.conj, p.e, p.pl, ldp, p.mag, ldm, p.sq);
    else
      oz_slice_cols<CX, false, ND><<<grid, 256, 0, s>>>(a.src, a.sb, a.lk, a.rows, K, a.conj, p.e, p.pl, ldp, p.mag, ldm, p.sq);
  }
  return cudaGetLastError();
}

template <int CX>
cudaError_t prepare(const Side& a, int K, int batch, const Planes& p, cudaStream_t s) {
  return p.mag ? prepare_digits<CX, 8>(a, K, batch, p, s) : prepare_digits<CX, 7>(a, K, batch, p, s);
}

// bf16 [n][rows][ldk] with K valid: digit planes in boxes of `digits` planes x
// `box` rows x 32 K, 64B swizzle, or (0) magnitudes in boxes of `box` rows x 64 K,
// 128B swizzle.
cudaError_t plane_map(CUtensorMap* map, const void* base, long n, long rows, int K, int ldk, int box, int digits) {
  static const PFN_cuTensorMapEncodeTiled_v12000 enc = [] {
    void* p = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault, &q) != cudaSuccess ||
        q != cudaDriverEntryPointSuccess)
      p = nullptr;
    return (PFN_cuTensorMapEncodeTiled_v12000)p;
  }();
  if (!enc) return cudaErrorNotSupported;
  cuuint64_t dims[3] = {(cuuint64_t)K, (cuuint64_t)rows, (cuuint64_t)n};
  cuuint64_t strides[2] = {(cuuint64_t)ldk * 2, (cuuint64_t)ldk * 2 * rows};
  cuuint32_t bx[3] = {(cuuint32_t)(digits ? TK : MK), (cuuint32_t)box, (cuuint32_t)(digits ? digits : 1)};
  cuuint32_t estr[3] = {1, 1, 1};
  return enc(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 3, (void*)base, dims, strides, bx, estr,
             CU_TENSOR_MAP_INTERLEAVE_NONE, digits ? CU_TENSOR_MAP_SWIZZLE_64B : CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
             CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS
             ? cudaSuccess
             : cudaErrorInvalidValue;
}

// One slab: the check (unless list is null), the digits, and what the check left.
template <int CX>
cudaError_t slab(const Side& l, const Side& n, int K, int nb, const Planes& pl, const Planes& pn, void* list, double* out,
                 long ldo, long sbo, bool pairs, double alpha, bool acc, const OzWork& w, cudaStream_t s) {
  const int Kr = K * CX, ldp = pad8i(Kr);
  OzShape g;
  g.lr = l.rows;
  g.nr = n.rows;
  g.lt = TL >> l.emb;
  g.nt = TN >> n.emb;
  g.mst = (K + MK - 1) / MK;
  g.nl = (int)plane_rows(l);
  g.nn = (int)plane_rows(n);
  g.nst = (Kr + TK - 1) / TK;
  g.tl = (int)tiles_of(l.rows, l.emb, TL);
  g.tn = (int)tiles_of(n.rows, n.emb, TN);
  g.lsh = l.emb;
  g.nsh = n.emb;
  g.el = l.rows;
  g.en = n.rows;
  g.ftn = g.tn;
  g.nd = list ? 8 : 7;
  g.units = (long)nb * g.tl * g.tn;
  g.pairs = pairs;
  g.acc = acc;
  g.alpha = alpha;
  g.ldo = ldo;
  g.sbo = sbo;
  if (g.units >= (1L << 31)) return cudaErrorInvalidValue;   // counted in 32 bits
  OzMaps maps, mags, wide;
  cudaError_t e = plane_map(&maps.n, pn.pl, (long)nb * g.nd, g.nn, Kr, ldp, TN, 7);
  if (e == cudaSuccess) e = plane_map(&maps.l, pl.pl, (long)nb * g.nd, g.nl, Kr, ldp, TL, 7);
  if (e == cudaSuccess && list) e = plane_map(&mags.n, pn.mag, nb, n.rows, K, pad8i(K), TN, 0);
  if (e == cudaSuccess && list) e = plane_map(&mags.l, pl.mag, nb, l.rows, K, pad8i(K), TL, 0);
  if (e == cudaSuccess && list) e = plane_map(&wide.n, pn.pl, (long)nb * g.nd, g.nn, Kr, ldp, WN, 8);
  if (e == cudaSuccess && list) e = plane_map(&wide.l, pl.pl, (long)nb * g.nd, g.nl, Kr, ldp, TL, 8);
  int dev = 0, nsm = 0;
  if (e == cudaSuccess) e = cudaGetDevice(&dev);
  if (e == cudaSuccess) e = cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev);
  constexpr size_t SMEM7 = Form<false>::SMEM, SMEM8 = Form<true>::SMEM;
  if (e == cudaSuccess)
    e = cudaFuncSetAttribute(oz_kernel<false>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)SMEM7);
  if (e == cudaSuccess && list)
    e = cudaFuncSetAttribute(oz_kernel<true>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)SMEM8);
  if (e == cudaSuccess && list)
    e = cudaFuncSetAttribute(oz_check_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)MSMEM);
  OzList f{};
  const unsigned grid = (unsigned)std::min<long>(g.units, nsm);
  if (!list) {
    if (e != cudaSuccess) return e;
    oz_kernel<false><<<grid, NT, SMEM7, s>>>(maps, g, pl.e, pn.e, out, f, w.err);
    if (w.launches) ++*w.launches;
    return cudaGetLastError();
  }
  f = list_at(list, g.units);
  if (e == cudaSuccess) e = cudaMemsetAsync(f.cnt, 0, 64 + sizeof(int) * (size_t)g.units, s);
  if (e != cudaSuccess) return e;
  oz_check_kernel<<<grid, MNT, MSMEM, s>>>(mags, g, pl.e, pn.e, pl.sq, pn.sq, f, w.err);
  oz_kernel<false><<<grid, NT, SMEM7, s>>>(maps, g, pl.e, pn.e, out, f, w.err);
  OzShape gw = g;
  gw.tn = (int)tiles_of(n.rows, n.emb, WN);
  gw.units = (long)nb * g.tl * gw.tn;
  if (gw.units >= (1L << 31)) return cudaErrorInvalidValue;
  oz_kernel<true><<<(unsigned)std::min<long>(gw.units, nsm), NT, SMEM8, s>>>(wide, gw, pl.e, pn.e, out, f, w.err);
  const Source sl{l.src, l.sb, l.lr, l.lk, l.conj}, sn{n.src, n.sb, n.lr, n.lk, n.conj};
  const unsigned xg = (unsigned)std::min<long>(2 * g.units, 2L * nsm);
  if constexpr (CX == 1)
    oz_exact_kernel<1, 4, 10><<<xg, 256, 0, s>>>(sl, sn, K, g, f, out, w.err);
  else if (pairs)
    oz_exact_kernel<2, 4, 5><<<xg, 256, 0, s>>>(sl, sn, K, g, f, out, w.err);
  else
    oz_exact_kernel<2, 2, 10><<<xg, 256, 0, s>>>(sl, sn, K, g, f, out, w.err);
  if (w.launches) *w.launches += 4;
  return cudaGetLastError();
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
  return g_limit < 0 ? w.bytes : std::min(w.bytes, (size_t)g_limit);
}

// Slabs of a product that fit in `room` bytes: batch entries, lane rows and
// column rows of each (of the sides' own rows).
struct Slabs {
  int bs, lrows, nrows;
};

// Whole batch entries where one fits, as many as take the fewest rounds of the
// SMs in all; else whole tiles of one entry: column tiles in up to half the room, lane tiles in what is left.
// Rows are rounded down to tiles, so that room for one tile of each side is
// enough and more of it never fails.
bool plan_slabs(int lrows, bool lemb, int nrows, bool nemb, int K, int CX, int batch, size_t room, Slabs& p) {
  auto need = [&](int nb, int l, int n) {
    return side_bytes(l, lemb, K, CX, nb) + side_bytes(n, nemb, K, CX, nb) +
           list_bytes(nb * tiles_of(l, lemb, TL) * tiles_of(n, nemb, TN));
  };
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
  const int bs = largest(batch, [&](int nb) { return need(nb, lrows, nrows) <= room; });
  if (bs > 0) {
    const long t = tiles_of(lrows, lemb, TL) * tiles_of(nrows, nemb, TN);
    auto rounds = [&](long n) { return (n * t + 151) / 152; };
    long best = -1;
    for (int n = bs; n > bs / 2; n--) {
      const long r = batch / n * rounds(n) + rounds(batch % n);
      if (best < 0 || r < best) {
        best = r;
        p.bs = n;
      }
    }
    return true;
  }
  const int lt = TL >> lemb, nt = TN >> nemb;   // rows of a tile
  auto lanes = [&](int t) { return (int)std::min<long>(lrows, (long)t * lt); };
  auto columns = [&](int t) { return (int)std::min<long>(nrows, (long)t * nt); };
  if (need(1, lanes(1), columns(1)) > room) return false;
  // (t: tiles in all, m: as many as fit; in as many slabs, but even ones)
  auto even = [](int t, int m) { const int parts = (t + m - 1) / m; return (t + parts - 1) / parts; };
  const int ct = (nrows + nt - 1) / nt, rt = (lrows + lt - 1) / lt;
  p.nrows = columns(even(ct, std::max(1, largest(ct, [&](int t) {
    return side_bytes(columns(t), nemb, K, CX, 1) <= room / 2 && need(1, lanes(1), columns(t)) <= room;
  }))));
  p.lrows = lanes(even(rt, largest(rt, [&](int t) { return need(1, lanes(t), p.nrows) <= room; })));
  return true;
}

// out(lane i, column j) over batch entries, in slabs that fit the scratch.
// pairs: the N side is embedded and out is complex [j / 2][i].  check: see the top.
template <int CX>
cudaError_t product(Side L, Side N, int K, int batch, double* out, long ldo, long sbo, bool pairs, double alpha,
                    bool acc, bool check, const OzWork& w, cudaStream_t s) {
  if (L.rows <= 0 || N.rows <= 0 || batch <= 0) return cudaSuccess;
  if (K <= 0 || (long)K * CX > OZ_MAX_K) return cudaErrorInvalidValue;   // the int64 sums stay below 2^62
  Slabs p;
  if (!plan_slabs(L.rows, L.emb, N.rows, N.emb, K, CX, batch, room_of(w), p)) return cudaErrorMemoryAllocation;
  const int bs = p.bs, lrows = p.lrows, nrows = p.nrows;
  for (int b0 = 0; b0 < batch; b0 += bs) {
    const int nb = std::min(bs, batch - b0);
    for (int n0 = 0; n0 < N.rows; n0 += nrows) {
      Side n = N;
      n.src += ((long)b0 * N.sb + (long)n0 * N.lr) * CX;
      n.rows = std::min(nrows, N.rows - n0);
      unsigned char* at = w.buf;
      Planes pn = planes_at(at, n.rows, n.emb, K, CX, nb);
      if (!check) pn.mag = nullptr;
      cudaError_t e = prepare<CX>(n, K, nb, pn, s);
      if (e != cudaSuccess) return e;
      if (w.launches) *w.launches += 2;
      at += side_bytes(n.rows, n.emb, K, CX, nb);
      for (int l0 = 0; l0 < L.rows; l0 += lrows) {
        Side l = L;
        l.src += ((long)b0 * L.sb + (long)l0 * L.lr) * CX;
        l.rows = std::min(lrows, L.rows - l0);
        Planes pl = planes_at(at, l.rows, l.emb, K, CX, nb);
        if (!check) pl.mag = nullptr;
        if ((e = prepare<CX>(l, K, nb, pl, s)) != cudaSuccess) return e;
        if (w.launches) *w.launches += 2;
        // pairs: double2 units along rows; embedded lanes: two doubles per complex column
        double* o = out + (pairs ? 2 * ((long)b0 * sbo + (long)n0 * ldo + l0)
                                 : (long)b0 * sbo + (long)n0 * ldo + (L.emb ? 2L : 1L) * l0);
        e = slab<CX>(l, n, K, nb, pl, pn, check ? at + side_bytes(l.rows, l.emb, K, CX, nb) : nullptr, o, ldo, sbo, pairs,
                     alpha, acc, w, s);
        if (e != cudaSuccess) return e;
      }
    }
  }
  return cudaSuccess;
}

}  // namespace

size_t oz_work_bytes(int M, int N, int K, int batch) {
  const bool ea = embed_a(M, N);
  return side_bytes(M, ea, K, 2, batch) + side_bytes(N, !ea, K, 2, batch) +
         list_bytes(batch * tiles_of(N, !ea, TL) * tiles_of(M, ea, TN));
}

size_t oz_work_min(int K) { return side_bytes(TN, false, K, 2, 1) + side_bytes(TL, false, K, 2, 1) + list_bytes(1); }

static bool plan(int M, int N, int K, int batch, bool real, size_t room, Slabs& p) {
  const bool ea = !real && embed_a(M, N);
  return plan_slabs(N, !real && !ea, M, ea, K, real ? 1 : 2, batch, room, p);
}

bool oz_fits(int M, int N, int K, int batch, bool real, const OzWork& w) {
  Slabs p;
  return w.buf && (real ? K : 2L * K) <= OZ_MAX_K && plan(M, N, K, batch, real, room_of(w), p);
}

void oz_limit(long long bytes) { g_limit = bytes; }

bool oz_plan(int M, int N, int K, int batch, bool real, size_t bytes, int out[3]) {
  Slabs p;
  const bool ok = plan(M, N, K, batch, real, bytes, p);
  out[0] = p.bs;
  out[1] = p.nrows;
  out[2] = p.lrows;
  return ok;
}

cudaError_t oz_alloc(OzWork& w, size_t want, size_t least, cudaStream_t s) {
  cudaError_t e = cudaErrorMemoryAllocation;
  unsigned char* p = nullptr;
  for (w.bytes = std::max(want, least);; w.bytes = std::max(least, w.bytes / 2)) {
    e = cudaMalloc((void**)&p, HEAD + w.bytes);
    if (e != cudaErrorMemoryAllocation) break;
    cudaGetLastError();
    if (w.bytes <= least) break;
  }
  if (e != cudaSuccess) {
    w = OzWork{};
    return e;
  }
  w.err = (int*)p;
  w.buf = p + HEAD;
  e = cudaMemsetAsync(p, 0, 64, s);
  if (e != cudaSuccess) oz_free(w);
  return e;
}

void oz_free(OzWork& w) {
  if (w.buf) cudaFree(w.buf - HEAD);
  w = OzWork{};
}

// The FP64 kernel takes 4.3 us per unit of K and round of its 64 x 64 tiles
// over the SMs (two multiply-adds a clock on each): 35 us for one tile of
// K = 8 (70 us measured for a stage of K = 8 to 16), and 0.3 ms for one of
// K = 71.  The digit form's eight launches are 45 us in all at K = 12, 55 to 65
// at K = 16 to 40.
bool oz_wins(int M, int N, int K, int batch) {
  const double tiles = ((M + 63) / 64) * (double)((N + 63) / 64) * batch;
  return ceil(tiles / 152.0) * K >= 10.0 && 2L * K <= OZ_MAX_K;
}

cudaError_t oz_gemm_z(int la, int lb, int M, int N, int K, const double2* A, int lda, long sA, const double2* B,
                      int ldb, long sB, double2* C, int ldc, long sC, int batch, bool check, const OzWork& w,
                      cudaStream_t s) {
  Side a{(const double*)A, M, la == A_KM ? 1L : (long)lda, la == A_KM ? (long)lda : 1L, sA, la == A_MK_CONJ, false};
  Side b{(const double*)B, N, lb == B_KN ? 1L : (long)ldb, lb == B_KN ? (long)ldb : 1L, sB, lb == B_NK_CONJ, false};
  if (embed_a(M, N)) {
    // embedded A as the columns, lanes along N: out[m][n] one double2 per lane
    a.emb = true;
    return product<2>(b, a, K, batch, (double*)C, ldc, sC, true, 1.0, false, check, w, s);
  }
  // embedded B as the lanes (real columns of the interleaved C), plain A rows as the columns
  b.emb = true;
  return product<2>(b, a, K, batch, (double*)C, 2L * ldc, 2 * sC, false, 1.0, false, check, w, s);
}

cudaError_t gemm_z_best(int la, int lb, int M, int N, int K, const double2* A, int lda, long sA, const double2* B,
                        int ldb, long sB, double2* C, int ldc, long sC, int batch, const OzWork& w, cudaStream_t s) {
  if (oz_wins(M, N, K, batch) && oz_fits(M, N, K, batch, false, w))
    return oz_gemm_z(la, lb, M, N, K, A, lda, sA, B, ldb, sB, C, ldc, sC, batch, true, w, s);
  if (w.launches) ++*w.launches;
  return gemm_z(la, lb, M, N, K, A, lda, sA, B, ldb, sB, C, ldc, sC, batch, s);
}

size_t oz_lane_bytes(int N, int K) { return exp_bytes(N, 1) + digit_bytes(N, false, K, 2, 1, 7); }
size_t oz_lanes_work(int M, int K) { return exp_bytes(M, 1) + digit_bytes(M, true, K, 2, 1, 7); }
bool oz_lanes_fit(int M, int K, const OzWork& w) { return w.buf && oz_lanes_work(M, K) <= room_of(w); }

static Planes unchecked(void* at, int rows, bool emb, int K) {
  Planes p = planes_at(at, rows, emb, K, 2, 1);
  p.mag = nullptr;
  return p;
}

cudaError_t oz_lane_prepare(const double2* B, int ldb, int N, int K, void* lanes, cudaStream_t s) {
  if (2L * K > OZ_MAX_K) return cudaErrorInvalidValue;
  const Side b{(const double*)B, N, 1L, (long)ldb, 0, false, false};
  return prepare<2>(b, K, 1, unchecked(lanes, N, false, K), s);
}

cudaError_t oz_gemm_z_lanes(int la, int M, int N, int K, const double2* A, int lda, void* lanes, double2* C, int ldc,
                            const OzWork& w, cudaStream_t s) {
  if (!oz_lanes_fit(M, K, w)) return cudaErrorMemoryAllocation;
  const Side a{(const double*)A, M, la == A_KM ? 1L : (long)lda, la == A_KM ? (long)lda : 1L, 0, la == A_MK_CONJ, true};
  const Side b{nullptr, N, 1L, 1L, 0, false, false};
  const Planes pa = unchecked(w.buf, M, true, K);
  const cudaError_t e = prepare<2>(a, K, 1, pa, s);
  if (e != cudaSuccess) return e;
  return slab<2>(b, a, K, 1, unchecked(lanes, N, false, K), pa, nullptr, (double*)C, ldc, 0, true, 1.0, false, w, s);
}

cudaError_t oz_gemm_d(bool a_km, bool b_kn, int M, int N, int K, const double* A, long lda, const double* B, long ldb,
                      double* C, long ldc, double alpha, bool acc, bool check, const OzWork& w, cudaStream_t s) {
  Side a{A, M, a_km ? 1L : lda, a_km ? lda : 1L, 0, false, false};
  Side b{B, N, b_kn ? 1L : ldb, b_kn ? ldb : 1L, 0, false, false};
  return product<1>(b, a, K, 1, C, ldc, 0, false, alpha, acc, check, w, s);
}
