// Pieces shared by the ISDF fit (isdf_fit.cu) and the adjoint of the fit in
// the orbital gradient (vo_grad.cu): the FP64 kernels of the fit's steps 1-3
// and the host-side geometry of a (grid, lattice, k mesh, points) problem.
#pragma once

#include "thc_internal.cuh"
#include "chol.cuh"
#include "oz_gemm.cuh"

#include <math.h>

#include <vector>

namespace {

constexpr int TB = 256;

unsigned blocks(long n) { return (unsigned)((n + TB - 1) / TB); }

// Ugc[P][f] = conj(U[f][pts[P]])
__global__ void gather_conj(const double2* __restrict__ U, int nf, long ng, const int* __restrict__ pts, int np,
                            double2* __restrict__ Ugc) {
  const long i = (long)blockIdx.x * TB + threadIdx.x;
  if (i >= (long)np * nf) return;
  const int P = (int)(i / nf), f = (int)(i % nf);
  const double2 u = U[(long)f * ng + pts[P]];
  Ugc[i] = make_double2(u.x, -u.y);
}

// R[i] = |B[i]|^2
__global__ void abs2_kernel(const double2* __restrict__ B, long n, double* __restrict__ R) {
  const long i = (long)blockIdx.x * TB + threadIdx.x;
  if (i >= n) return;
  const double2 b = B[i];
  R[i] = b.x * b.x + b.y * b.y;
}

// S[P][Q] = R[P][pts[Q]]
__global__ void gather_cols(const double* __restrict__ R, long ng, const int* __restrict__ pts, int np,
                            double* __restrict__ S) {
  const long i = (long)blockIdx.x * TB + threadIdx.x;
  if (i >= (long)np * np) return;
  const int P = (int)(i / np), Q = (int)(i % np);
  S[i] = R[(long)P * ng + pts[Q]];
}

// X = L^-T L^-1 X for every column r of X[n][ng], in place.
__global__ void chol_solve(const double* __restrict__ L, double* __restrict__ X, int n, long ng) {
  const long r = (long)blockIdx.x * TB + threadIdx.x;
  if (r >= ng) return;
  for (int j = 0; j < n; j++) {
    double a = X[(long)j * ng + r];
    for (int t = 0; t < j; t++) a -= L[(long)j * n + t] * X[(long)t * ng + r];
    X[(long)j * ng + r] = a / L[(long)j * n + j];
  }
  for (int j = n - 1; j >= 0; j--) {
    double a = X[(long)j * ng + r];
    for (int t = j + 1; t < n; t++) a -= L[(long)t * n + j] * X[(long)t * ng + r];
    X[(long)j * ng + r] = a / L[(long)j * n + j];
  }
}

// One axis of the forward DFT of [np][g1][g2][g3]: out = sum_j in(j) tw[(j m) mod g].
// `real_in` reads a real array (the vectors themselves) for the first axis.
__global__ void dft_axis_kernel(const void* __restrict__ in, bool real_in, double2* __restrict__ out, long total,
                                int g, long st, const double2* __restrict__ tw) {
  const long i = (long)blockIdx.x * TB + threadIdx.x;
  if (i >= total) return;
  const int m = (int)((i / st) % g);
  const long base = i - (long)m * st;
  double re = 0.0, im = 0.0;
  for (int j = 0, jm = 0; j < g; j++, jm = (jm + m) % g) {
    const double2 w = tw[jm];
    if (real_in) {
      const double x = ((const double*)in)[base + (long)j * st];
      re += x * w.x;
      im += x * w.y;
    } else {
      const double2 x = ((const double2*)in)[base + (long)j * st];
      re += x.x * w.x - x.y * w.y;
      im += x.x * w.y + x.y * w.x;
    }
  }
  out[i] = make_double2(re, im);
}

// The same axis by a mixed-radix (Stockham) FFT in shared memory, for lengths
// whose primes are 2, 3, 5 and 7: the direct sum's 4 g FP64 multiply-adds per
// element (160 at g = 40, 38 ms for the three axes of 600 vectors on a 40^3
// grid, bound by the FP64 pipe) become about 35.  A block takes FW lines that
// lie side by side: lines FW st apart for the contiguous axis, else columns of
// the slab of one (outer, inner) index range.
constexpr int FW = 16;
struct FftPlan {
  int g, nr;
  int r[8];
};

// Radices 4, 2, 3, 5, 7 of g; nr = 0 where other primes are left.
inline FftPlan fft_plan(int g) {
  FftPlan p{};
  p.g = g;
  int m = g;
  for (int r : {4, 2, 3, 5, 7})
    while (m % r == 0 && p.nr < 8) {
      p.r[p.nr++] = r;
      m /= r;
    }
  if (m != 1 || g > 256) p.nr = 0;
  return p;
}

// The r-point DFT of v (e^{-2 pi i / r}); w: the twiddles e^{-2 pi i t / g}, stride g / r.
template <int R>
__device__ __forceinline__ void dft_small(double2* v, const double2* __restrict__ w, int stride) {
  if constexpr (R == 2) {
    const double2 a = v[0];
    v[0] = cadd(a, v[1]);
    v[1] = csub(a, v[1]);
  } else if constexpr (R == 4) {
    const double2 a = cadd(v[0], v[2]), b = csub(v[0], v[2]), c = cadd(v[1], v[3]), d = csub(v[1], v[3]);
    v[0] = cadd(a, c);
    v[2] = csub(a, c);
    v[1] = make_double2(b.x + d.y, b.y - d.x);
    v[3] = make_double2(b.x - d.y, b.y + d.x);
  } else {
    // odd R: pairs t, R - t share a twiddle's real part and its imaginary part up to sign
    constexpr int H = R / 2;
    double2 s[H], d[H], z = v[0];
#pragma unroll
    for (int t = 0; t < H; t++) {
      s[t] = cadd(v[t + 1], v[R - 1 - t]);
      d[t] = csub(v[t + 1], v[R - 1 - t]);
    }
#pragma unroll
    for (int t = 0; t < H; t++) z = cadd(z, s[t]);
    double2 o[R];
#pragma unroll
    for (int q = 1; q <= H; q++) {
      double2 a = v[0], b = make_double2(0.0, 0.0);
#pragma unroll
      for (int t = 0; t < H; t++) {
        const double2 c = w[((t + 1) * q % R) * stride];
        a.x = fma(c.x, s[t].x, a.x);
        a.y = fma(c.x, s[t].y, a.y);
        b.x = fma(-c.y, d[t].y, b.x);
        b.y = fma(c.y, d[t].x, b.y);
      }
      o[q] = cadd(a, b);
      o[R - q] = csub(a, b);
    }
    v[0] = z;
#pragma unroll
    for (int q = 1; q < R; q++) v[q] = o[q];
  }
}

template <int R>
__device__ __forceinline__ void fft_stage(const double2* x, double2* y, int g, int ns, const double2* __restrict__ tw) {
  const int m = g / R, step = g / (ns * R);
  for (int t = threadIdx.x; t < m * FW; t += TB) {
    const int w = t % FW, i = t / FW, k = i % ns;
    double2 v[R];
#pragma unroll
    for (int q = 0; q < R; q++) {
      v[q] = x[(i + q * m) * FW + w];
      if (q > 0 && ns > 1) v[q] = cmul(v[q], tw[q * k * step]);
    }
    dft_small<R>(v, tw, m);
    const int o = (i / ns) * ns * R + k;
#pragma unroll
    for (int q = 0; q < R; q++) y[(o + q * ns) * FW + w] = v[q];
  }
}

__global__ void __launch_bounds__(TB) fft_axis_kernel(const void* __restrict__ in, bool real_in,
                                                      double2* __restrict__ out, long lines, long st, FftPlan p,
                                                      const double2* __restrict__ tw) {
  extern __shared__ double2 fsm[];
  const int g = p.g;
  double2 *x = fsm, *y = fsm + g * FW, *stw = fsm + 2 * g * FW;
  for (int t = threadIdx.x; t < g; t += TB) stw[t] = tw[t];
  // line n: base (n / st) st g + n % st, elements st apart
  const long n0 = (long)blockIdx.x * FW;
  for (int t = threadIdx.x; t < g * FW; t += TB) {
    // the contiguous axis is read along its lines, the others across them
    const int w = st == 1 ? t / g : t % FW, j = st == 1 ? t % g : t / FW;
    const long n = n0 + w;
    double2 v = make_double2(0.0, 0.0);
    if (n < lines) {
      const long o = (n / st) * st * g + n % st + (long)j * st;
      if (real_in) v.x = ((const double*)in)[o];
      else v = ((const double2*)in)[o];
    }
    x[j * FW + w] = v;
  }
  int ns = 1;
  for (int s = 0; s < p.nr; s++) {
    __syncthreads();
    switch (p.r[s]) {
      case 2: fft_stage<2>(x, y, g, ns, stw); break;
      case 3: fft_stage<3>(x, y, g, ns, stw); break;
      case 4: fft_stage<4>(x, y, g, ns, stw); break;
      case 5: fft_stage<5>(x, y, g, ns, stw); break;
      default: fft_stage<7>(x, y, g, ns, stw); break;
    }
    ns *= p.r[s];
    double2* z = x;
    x = y;
    y = z;
  }
  __syncthreads();
  for (int t = threadIdx.x; t < g * FW; t += TB) {
    const int w = st == 1 ? t / g : t % FW, j = st == 1 ? t % g : t / FW;
    const long n = n0 + w;
    if (n < lines) out[(n / st) * st * g + n % st + (long)j * st] = x[j * FW + w];
  }
}

// One axis (length g, stride st) of the forward DFT of `total` values; fft = false: by direct sums.
inline cudaError_t dft_axis(const void* in, bool real_in, double2* out, long total, int g, long st,
                            const double2* tw, cudaStream_t s, bool fft = true) {
  const FftPlan p = fft_plan(g);
  const long lines = total / g;
  if (fft && p.nr > 0 && lines < (1L << 34)) {
    const size_t sm = sizeof(double2) * (size_t)g * (2 * FW + 1);
    const cudaError_t e = cudaFuncSetAttribute(fft_axis_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
    if (e != cudaSuccess) return e;
    fft_axis_kernel<<<(unsigned)((lines + FW - 1) / FW), TB, sm, s>>>(in, real_in, out, lines, st, p, tw);
  } else {
    dft_axis_kernel<<<blocks(total), TB, 0, s>>>(in, real_in, out, total, g, st, tw);
  }
  return cudaGetLastError();
}

// Minimum-image fractional representatives of q = qco / mesh along one axis.
std::vector<double> axis_reps(int qc, int n) {
  const double f = (double)(((qc % n) + n) % n) / n;
  if (fabs(f - 0.5) < 1e-12) return {0.5, -0.5};
  if (f > 0.5) return {f - 1.0};
  return {f};
}


// Reciprocal rows b_i with a_i . b_j = 2 pi delta_ij.
struct Recip {
  double b[9];   // rows b1, b2, b3
};

// The geometry of one fit: grid and mesh sizes, cell volume, reciprocal rows,
// the G set without Nyquist planes (integer coordinates and the flat grid
// index of each), the Cartesian point positions, and the per-axis twiddles
// e^{-2 pi i t / g} (axis a's at tw[off[a]]).
struct FitGeom {
  int g[3], n[3];
  long ng;
  int nk;
  double vol;
  Recip B;
  std::vector<int> gm, flat;
  std::vector<double> rP;
  std::vector<double2> tw;
  int off[3];
};

// Checks the arguments a fit shares (grid sizes >= 1, mesh sizes in 1..8,
// 1 <= npts <= N_g distinct grid indices, a cell of positive volume) and fills
// `geo`; false on a bad one.
inline bool fit_geometry(const int* grid_host, const double* lattice_host, const int* mesh_host,
                         const int* points_host, int npts, FitGeom& geo) {
  const int g1 = grid_host[0], g2 = grid_host[1], g3 = grid_host[2];
  const int n1 = mesh_host[0], n2 = mesh_host[1], n3 = mesh_host[2];
  if (g1 < 1 || g2 < 1 || g3 < 1 || n1 < 1 || n2 < 1 || n3 < 1 || n1 > 8 || n2 > 8 || n3 > 8) return false;
  const long ng = (long)g1 * g2 * g3;
  if (npts < 1 || npts > ng) return false;
  std::vector<char> seen(ng, 0);
  for (int P = 0; P < npts; P++) {
    const int p = points_host[P];
    if (p < 0 || p >= ng || seen[p]) return false;   // points must be distinct grid indices
    seen[p] = 1;
  }
  const double* a = lattice_host;
  const double det = a[0] * (a[4] * a[8] - a[5] * a[7]) - a[1] * (a[3] * a[8] - a[5] * a[6]) +
                     a[2] * (a[3] * a[7] - a[4] * a[6]);
  const double vol = fabs(det);
  if (!(vol > 0)) return false;
  geo.g[0] = g1, geo.g[1] = g2, geo.g[2] = g3;
  geo.n[0] = n1, geo.n[1] = n2, geo.n[2] = n3;
  geo.ng = ng;
  geo.nk = n1 * n2 * n3;
  geo.vol = vol;
  {
    const double c = 2.0 * M_PI / det;
    const double* a1 = a;
    const double* a2 = a + 3;
    const double* a3 = a + 6;
    auto cross = [](const double* x, const double* y, double* o) {
      o[0] = x[1] * y[2] - x[2] * y[1];
      o[1] = x[2] * y[0] - x[0] * y[2];
      o[2] = x[0] * y[1] - x[1] * y[0];
    };
    cross(a2, a3, geo.B.b);
    cross(a3, a1, geo.B.b + 3);
    cross(a1, a2, geo.B.b + 6);
    for (double& x : geo.B.b) x *= c;
  }
  const int h1 = (g1 - 1) / 2, h2 = (g2 - 1) / 2, h3 = (g3 - 1) / 2;
  geo.gm.clear();
  geo.flat.clear();
  for (int i = -h1; i <= h1; i++)
    for (int j = -h2; j <= h2; j++)
      for (int l = -h3; l <= h3; l++) {
        geo.gm.push_back(i);
        geo.gm.push_back(j);
        geo.gm.push_back(l);
        geo.flat.push_back((((i % g1) + g1) % g1 * g2 + ((j % g2) + g2) % g2) * g3 + ((l % g3) + g3) % g3);
      }
  geo.rP.assign(3 * (size_t)npts, 0.0);
  for (int P = 0; P < npts; P++) {
    const int p = points_host[P];
    const double f0 = (double)(p / (g2 * g3)) / g1, f1 = (double)((p / g3) % g2) / g2, f2 = (double)(p % g3) / g3;
    for (int x = 0; x < 3; x++) geo.rP[3 * P + x] = f0 * a[x] + f1 * a[3 + x] + f2 * a[6 + x];
  }
  geo.tw.assign(g1 + g2 + g3, make_double2(0.0, 0.0));
  geo.off[0] = 0, geo.off[1] = g1, geo.off[2] = g1 + g2;
  const int gs[3] = {g1, g2, g3};
  for (int ax = 0; ax < 3; ax++)
    for (int t = 0; t < gs[ax]; t++) {
      const double ang = -2.0 * M_PI * t / gs[ax];
      geo.tw[geo.off[ax] + t] = make_double2(cos(ang), sin(ang));
    }
  return true;
}

// The device memory of one call.  The scratch of its digit products is
// optional (without it they run on the FP64 pipe): an allocation that the device
// has no room for is tried again once the scratch is given back.
struct DeviceMemory {
  OzWork oz;
  int lost = 0;                       // error word of scratch given back
  int fail_at = take_fail_alloc();    // test hook: index of the allocation that fails the first time
  int n = 0;

  template <typename T>
  cudaError_t get(T** p, size_t bytes) {
    cudaError_t e = n++ == fail_at ? cudaErrorMemoryAllocation : cudaMalloc((void**)p, bytes);
    if (e != cudaErrorMemoryAllocation) return e;
    cudaGetLastError();
    *p = nullptr;
    if (!oz.buf) return e;
    e = cudaDeviceSynchronize();
    if (e == cudaSuccess) e = wait_error(&lost);
    oz_free(oz);
    return e == cudaSuccess ? cudaMalloc((void**)p, bytes) : e;
  }

  // Whether a wait of a digit product gave up (nonzero), of the work complete so far.
  cudaError_t wait_error(int* h) {
    *h = lost;
    if (!oz.buf) return cudaSuccess;
    int now = 0;
    const cudaError_t e = cudaMemcpy(&now, oz.err, sizeof(int), cudaMemcpyDeviceToHost);
    *h |= now;
    return e;
  }

  // Scratch of a fit and of its adjoint: the whole operands of the metric and of
  // the products of depth kdeep (over the grid or its G set, npts x ndeep; 0:
  // none), up to 1.25 GB (larger slabs measured no faster for the metric), at
  // least what the metric's least slab needs.  deep: the deep products are to be
  // whole where eight times as much is free, up to 8 GB (their slabs hold a few
  // tiles each and take the time of a whole product one after the other: FP64
  // contraction at 3 x 3 x 3 k, N_P = 600, 40^3 grid, 2939 ms in 1.25 GB, 280 whole).
  cudaError_t scratch(int npts, long ng, int nfunc, int ndeep, int kdeep, bool deep, cudaStream_t s) {
    const size_t least = oz_work_min(nfunc);
    size_t want = std::max(oz_work_bytes(npts, (int)ng, nfunc, 1), oz_work_bytes(npts, (int)ng, npts, 1));
    if (ndeep > 0) want = std::max(want, std::max(oz_work_min(kdeep), oz_work_bytes(npts, ndeep, kdeep, 1)));
    size_t most = (size_t)5 << 28, room = 0, total = 0;
    if (deep && cudaMemGetInfo(&room, &total) == cudaSuccess) most = std::max(most, std::min(room / 8, (size_t)8 << 30));
    const cudaError_t e = oz_alloc(oz, std::max(least, std::min(want, most)), least, s);
    if (e != cudaErrorMemoryAllocation) return e;
    cudaGetLastError();
    return cudaSuccess;
  }
};

}  // namespace
