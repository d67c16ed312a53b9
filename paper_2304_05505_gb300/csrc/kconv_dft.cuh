// The separable 3-D DFT of one element's values over the k mesh, axis by axis
// with radix-2/3/4 butterflies (6 by Good-Thomas) or a direct DFT, shared by
// the forms of the k-convolution.
#pragma once

#include "thc_internal.cuh"

#include <math.h>

namespace {

constexpr int MAXL = 8;

struct Twiddles {
  int n[3];
  double c[3][MAXL], s[3][MAXL];      // cos, sin of 2 pi r / n_ax
  float ch[3][MAXL], cl[3][MAXL];     // FP32 hi/lo split of c
  float sh[3][MAXL], sl[3][MAXL];
};

template <typename R> struct Tw;
template <> struct Tw<double> {
  __device__ static double2 mul(double2 v, const Twiddles& t, int ax, int r, int sign) {
    double c = t.c[ax][r], s = sign * t.s[ax][r];
    return make_double2(v.x * c - v.y * s, v.x * s + v.y * c);
  }
  __device__ static double2 mul_s3(double2 d, int sign) {
    // i * sign * sqrt(3)/2 * d
    const double h = 0.86602540378443864676;
    return make_double2(-sign * h * d.y, sign * h * d.x);
  }
};
template <> struct Tw<float> {
  __device__ static float2 mul(float2 v, const Twiddles& t, int ax, int r, int sign) {
    float ch = t.ch[ax][r], cl = t.cl[ax][r];
    float sh = sign * t.sh[ax][r], sl = sign * t.sl[ax][r];
    float re = fmaf(v.x, ch, -v.y * sh) + (v.x * cl - v.y * sl);
    float im = fmaf(v.x, sh, v.y * ch) + (v.x * sl + v.y * cl);
    return make_float2(re, im);
  }
  __device__ static float2 mul_s3(float2 d, int sign) {
    const float hh = 0.866025388240814208984375f;       // float(sqrt(3)/2)
    const float hl = 1.5543625e-8f;                     // sqrt(3)/2 - hh
    float re = -(d.y * hh + d.y * hl);
    float im = d.x * hh + d.x * hl;
    return make_float2(sign * re, sign * im);
  }
};

// (S: int, or long where the values of an element lie an N_P^2 apart)
template <typename R, int L, typename S>
__device__ __forceinline__ void line_dft(typename cplx<R>::type* x, S step, const Twiddles& tw,
                                         int ax, int sign) {
  typedef typename cplx<R>::type CT;
  CT v[L];
#pragma unroll
  for (int j = 0; j < L; j++) v[j] = x[j * step];
  if constexpr (L == 2) {
    x[0] = cadd(v[0], v[1]);
    x[step] = csub(v[0], v[1]);
  } else if constexpr (L == 3) {
    CT t = cadd(v[1], v[2]);
    CT d = csub(v[1], v[2]);
    CT m = CT{v[0].x - (R)0.5 * t.x, v[0].y - (R)0.5 * t.y};
    CT s = Tw<R>::mul_s3(d, sign);
    x[0] = cadd(v[0], t);
    x[step] = cadd(m, s);
    x[2 * step] = csub(m, s);
  } else if constexpr (L == 4) {
    CT a0 = cadd(v[0], v[2]), a1 = csub(v[0], v[2]);
    CT b0 = cadd(v[1], v[3]), b1 = csub(v[1], v[3]);
    CT ib1 = CT{-sign * b1.y, sign * b1.x};   // i * sign * b1
    x[0] = cadd(a0, b0);
    x[2 * step] = csub(a0, b0);
    x[step] = cadd(a1, ib1);
    x[3 * step] = csub(a1, ib1);
  } else if constexpr (L == 6) {
    // prime-factor (Good-Thomas) 6 = 2 x 3, no twiddles between the factors:
    // inputs n = (3 n1 + 2 n2) mod 6, outputs m = (3 m1 + 4 m2) mod 6,
    // X[m] = sum_{n1} (-1)^{n1 m1} sum_{n2} x[n] w3^{n2 m2}
    CT y0[3], y1[3];
    auto dft3v = [&](CT a, CT b, CT c, CT* y) {
      const CT t = cadd(b, c), d = csub(b, c);
      const CT m = CT{a.x - (R)0.5 * t.x, a.y - (R)0.5 * t.y};
      const CT sd = Tw<R>::mul_s3(d, sign);
      y[0] = cadd(a, t);
      y[1] = cadd(m, sd);
      y[2] = csub(m, sd);
    };
    dft3v(v[0], v[2], v[4], y0);
    dft3v(v[3], v[5], v[1], y1);
    x[0] = cadd(y0[0], y1[0]);
    x[3 * step] = csub(y0[0], y1[0]);
    x[4 * step] = cadd(y0[1], y1[1]);
    x[step] = csub(y0[1], y1[1]);
    x[2 * step] = cadd(y0[2], y1[2]);
    x[5 * step] = csub(y0[2], y1[2]);
  } else {
#pragma unroll
    for (int m = 0; m < L; m++) {
      CT acc = v[0];
#pragma unroll
      for (int j = 1; j < L; j++) acc = cadd(acc, Tw<R>::mul(v[j], tw, ax, (j * m) % L, sign));
      x[m * step] = acc;
    }
  }
}

template <typename R, typename S>
__device__ void dft_axis(typename cplx<R>::type* x, S T, const Twiddles& tw, int ax, int sign) {
  const int n1 = tw.n[0], n2 = tw.n[1], n3 = tw.n[2];
  const int L = tw.n[ax];
  if (L == 1) return;
  int nout, sout, nin, sin_, step;
  if (ax == 0) { nout = n2; sout = n3; nin = n3; sin_ = 1; step = n2 * n3; }
  else if (ax == 1) { nout = n1; sout = n2 * n3; nin = n3; sin_ = 1; step = n3; }
  else { nout = n1; sout = n2 * n3; nin = n2; sin_ = n3; step = 1; }
  for (int o = 0; o < nout; o++)
    for (int i = 0; i < nin; i++) {
      typename cplx<R>::type* base = x + (long)(o * sout + i * sin_) * T;
      const S st = step * T;
      switch (L) {
        case 2: line_dft<R, 2>(base, st, tw, ax, sign); break;
        case 3: line_dft<R, 3>(base, st, tw, ax, sign); break;
        case 4: line_dft<R, 4>(base, st, tw, ax, sign); break;
        case 5: line_dft<R, 5>(base, st, tw, ax, sign); break;
        case 6: line_dft<R, 6>(base, st, tw, ax, sign); break;
        case 7: line_dft<R, 7>(base, st, tw, ax, sign); break;
        default: line_dft<R, 8>(base, st, tw, ax, sign); break;
      }
    }
}

// The DFT over the mesh of the values x[a T], a on the mesh index.
template <typename R, typename S>
__device__ __forceinline__ void dft3(typename cplx<R>::type* x, S T, const Twiddles& tw, int sign) {
  dft_axis<R>(x, T, tw, 0, sign);
  dft_axis<R>(x, T, tw, 1, sign);
  dft_axis<R>(x, T, tw, 2, sign);
}

Twiddles make_twiddles(int n1, int n2, int n3) {
  Twiddles t;
  t.n[0] = n1; t.n[1] = n2; t.n[2] = n3;
  for (int ax = 0; ax < 3; ax++)
    for (int r = 0; r < MAXL; r++) {
      int L = t.n[ax];
      double c = 1.0, s = 0.0;
      if (r < L && L > 0) {
        // exact values at multiples of pi/2
        if ((4 * r) % L == 0) {
          int q = (4 * r) / L;   // quarter turns
          c = (q == 0) ? 1.0 : (q == 2) ? -1.0 : 0.0;
          s = (q == 1) ? 1.0 : (q == 3) ? -1.0 : 0.0;
        } else {
          c = cos(2.0 * M_PI * r / L);
          s = sin(2.0 * M_PI * r / L);
        }
      }
      t.c[ax][r] = c;
      t.s[ax][r] = s;
      t.ch[ax][r] = (float)c;
      t.cl[ax][r] = (float)(c - (double)t.ch[ax][r]);
      t.sh[ax][r] = (float)s;
      t.sl[ax][r] = (float)(s - (double)t.sh[ax][r]);
    }
  return t;
}

}  // namespace
