// Interpolation-point selection (setup, not part of the timed build):
// greedy pivoted Cholesky, in FP64, of the Gram matrix of occupied pair
// products
//   A(r, r') = | sum_f conj(U[f][r]) U[f][r'] |^2,   f = (k, i), U[f][r] = u^k_i(r)
// (the metric of the least-squares fit of Eq. pbcinterpvec restricted to
// occupied orbitals, Eq. orbprodoo).  Pivoted Cholesky picks the same points
// as the QR decomposition with column pivoting of Sec. 2.1 in exact
// arithmetic.  A is never formed: each step builds one column from U.
//
// Per step j (host loop):
//   argmax  p = argmax_r d[r] (lowest r among equal values), d[p], sum_r d[r]
//           (block partials, then one block)
//   column  a = |B(:, p)|^2, l = (a - sum_{t<j} L[t][:] L[t][p]) / sqrt(d[p]),
//           L[j][:] = l, d = max(d - l^2, 0), d[p] = 0; a block takes 32
//           candidates (one per lane, coalesced) and its 8 warps split the
//           sums over f and over t, added in a fixed order
// The loop stops after npts pivots or when sum d <= rel_tol * trace(A).
//
// That takes one pass over U and nfunc * ncand complex FP64 multiply-adds per
// pivot: 1.28 ms each at 1620 functions on a 40^3 grid, at the FP64 pipe's
// rate.  Larger selections therefore go in blocks of up to 40 pivots:
//   1. the set S of up to 800 candidates with the largest residuals: all with
//      d at or above the edge of a histogram bin (1/256 of an octave wide)
//   2. the residual matrix on S, |B|^2 minus the earlier rows' products, with
//      both products from digits on the tensor cores (oz_gemm.cu)
//   3. pivots from S by the same rule, one block, as long as the largest
//      residual in S is at or above that edge: the residuals outside S are
//      below it and never grow, so these are the pivots of the whole set
//   4. the block's columns for all candidates: one product with the digits of
//      U, which are made once, one with the earlier rows of L, and a kernel
//      that finishes the block's own triangle, d and sum d after every pivot
// The products are not checked entry by entry (oz_gemm.cu); what the selection
// needs of A(p, c) is its error relative to sqrt(A(p, p) A(c, c)), and digits
// hold that to 2^-8 of what FP64 sums may leave.  |u| of a candidate is at most
// A(c, c)^(1/4) and |L[s][c]| at most sqrt(A(c, c)), so B errs by at most 4 K 2^-62
// (A(p, p) A(c, c))^(1/4), for K functions, and the sum over j earlier rows by
// 2 j 2^-62 sqrt(A(p, p) A(c, c)).  With d_c <= d_p that reaches the residual of c
// as 2 l dl <= (8 K + 2 j) 2^-61 sqrt(A(p, p) / d_p) of A(c, c).  (With the check
// the rows of points far apart, which have no entry in common, ran in FP64: 93
// ms at 600 points, the residuals as far from 64 bits as without, 4.5e-12.)
// (767 ms to 49 ms for 600 points.)  Where S comes out empty (more than 800
// candidates within a bin of the largest), or a block ends after so few pivots
// that they are cheaper one by one, pivots are taken the first way: 8 of them
// before the next block, twice as many each time until a block pays again (200
// points of equal density among 2400 at 420 functions: 48 to 12 ms).
#include "oz_gemm.cuh"
#include "thc_internal.cuh"

#include <stddef.h>

#include <algorithm>

namespace {

constexpr int PT = 256;

__global__ void diag_kernel(const double2* __restrict__ U, int nfunc, int ncand, double* __restrict__ d) {
  const int c = blockIdx.x * blockDim.x + threadIdx.x;
  if (c >= ncand) return;
  double rho = 0.0;
  for (int f = 0; f < nfunc; f++) {
    const double2 u = U[(long)f * ncand + c];
    rho += u.x * u.x + u.y * u.y;
  }
  d[c] = rho * rho;
}

struct Best {
  double v;
  int i;
};

__device__ __forceinline__ Best better(Best a, Best b) {
  if (b.v > a.v || (b.v == a.v && b.i < a.i)) return b;
  return a;
}

// Block partials of (max d, its lowest index) and of sum d.
__global__ void __launch_bounds__(PT) argmax_partial(const double* __restrict__ d, int n, double* pv, int* pi,
                                                     double* ps) {
  __shared__ double sv[PT];
  __shared__ int si[PT];
  __shared__ double ss[PT];
  Best b{-1.0, 0x7fffffff};
  double s = 0.0;
  for (int c = blockIdx.x * PT + threadIdx.x; c < n; c += gridDim.x * PT) {
    b = better(b, Best{d[c], c});
    s += d[c];
  }
  sv[threadIdx.x] = b.v;
  si[threadIdx.x] = b.i;
  ss[threadIdx.x] = s;
  __syncthreads();
  for (int o = PT / 2; o > 0; o >>= 1) {
    if (threadIdx.x < o) {
      Best x = better(Best{sv[threadIdx.x], si[threadIdx.x]}, Best{sv[threadIdx.x + o], si[threadIdx.x + o]});
      sv[threadIdx.x] = x.v;
      si[threadIdx.x] = x.i;
      ss[threadIdx.x] += ss[threadIdx.x + o];
    }
    __syncthreads();
  }
  if (threadIdx.x == 0) {
    pv[blockIdx.x] = sv[0];
    pi[blockIdx.x] = si[0];
    ps[blockIdx.x] = ss[0];
  }
}

// One block: final (p, d[p], trace) into sel (int) and selv[0..1].
__global__ void __launch_bounds__(PT) argmax_final(const double* pv, const int* pi, const double* ps, int nb,
                                                   int* sel, double* selv) {
  __shared__ double sv[PT];
  __shared__ int si[PT];
  __shared__ double ss[PT];
  Best b{-1.0, 0x7fffffff};
  double s = 0.0;
  for (int i = threadIdx.x; i < nb; i += PT) {
    b = better(b, Best{pv[i], pi[i]});
    s += ps[i];
  }
  sv[threadIdx.x] = b.v;
  si[threadIdx.x] = b.i;
  ss[threadIdx.x] = s;
  __syncthreads();
  for (int o = PT / 2; o > 0; o >>= 1) {
    if (threadIdx.x < o) {
      Best x = better(Best{sv[threadIdx.x], si[threadIdx.x]}, Best{sv[threadIdx.x + o], si[threadIdx.x + o]});
      sv[threadIdx.x] = x.v;
      si[threadIdx.x] = x.i;
      ss[threadIdx.x] += ss[threadIdx.x + o];
    }
    __syncthreads();
  }
  if (threadIdx.x == 0) {
    sel[0] = si[0];
    selv[0] = sv[0];
    selv[1] = ss[0];
  }
}

constexpr int CW = 8;   // warps of a column block

__global__ void __launch_bounds__(32 * CW) column_kernel(const double2* __restrict__ U, int nfunc, int ncand, int j,
                                                         const int* __restrict__ sel,
                                                         const double* __restrict__ selv, double* __restrict__ L,
                                                         double* __restrict__ d) {
  __shared__ double sr[CW][32], si[CW][32], sl[CW][32];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const int c = blockIdx.x * 32 + lane;
  const int p = sel[0];
  double br = 0.0, bi = 0.0, ll = 0.0;   // B(c, p) = sum_f conj(U[f][c]) U[f][p]; sum_t L[t][c] L[t][p]
  if (c < ncand) {
    for (int f = w; f < nfunc; f += CW) {
      const double2 u = U[(long)f * ncand + c];
      const double2 v = U[(long)f * ncand + p];
      br += u.x * v.x + u.y * v.y;
      bi += u.x * v.y - u.y * v.x;
    }
    for (int t = w; t < j; t += CW) ll += L[(long)t * ncand + c] * L[(long)t * ncand + p];
  }
  sr[w][lane] = br;
  si[w][lane] = bi;
  sl[w][lane] = ll;
  __syncthreads();
  if (w != 0 || c >= ncand) return;
  for (int k = 1; k < CW; k++) {
    br += sr[k][lane];
    bi += si[k][lane];
    ll += sl[k][lane];
  }
  const double l = (br * br + bi * bi - ll) / sqrt(selv[0]);
  L[(long)j * ncand + c] = l;
  d[c] = (c == p) ? 0.0 : fmax(d[c] - l * l, 0.0);
}

// ---------------------------------------------------------------------------
// blocks of pivots
// ---------------------------------------------------------------------------

constexpr int MS = 800;        // candidates of a block's set (its matrix: 130 output tiles, one round of the SMs)
constexpr int TP = 40;         // pivots of a block (80 embedded columns, one tile)
constexpr int NBIN = 64 * 256;
constexpr int FT = 128;        // threads of finish_kernel

// Bin of a residual: 256 per octave, 64 octaves down from the largest; 0 for none.
__device__ __forceinline__ int bin_of(double v, double top) {
  if (!(v > 0.0)) return 0;
  const int h = __double2hiint(v), e = 63 - ((__double2hiint(top) >> 20) - (h >> 20));
  return e < 0 ? 0 : e * 256 + ((h >> 12) & 255);
}

__global__ void __launch_bounds__(PT) hist_kernel(const double* __restrict__ d, int n, const double* __restrict__ selv,
                                                  int* __restrict__ hist) {
  const double top = selv[0];
  for (int c = blockIdx.x * PT + threadIdx.x; c < n; c += gridDim.x * PT) {
    const int b = bin_of(d[c], top);
    if (b > 0) atomicAdd(hist + b, 1);
  }
}

// The set: edge[0] = the lowest bin with at most MS candidates in it and above;
// idx = those candidates, ascending, then -1; edge[1] their count.  One block of 1024.
__global__ void __launch_bounds__(1024) pick_kernel(const double* __restrict__ d, int n,
                                                    const double* __restrict__ selv, const int* __restrict__ hist,
                                                    int* __restrict__ idx, int* __restrict__ edge) {
  __shared__ int ws[33], kb;
  const int t = threadIdx.x, lane = t & 31, w = t >> 5;
  // bins from the top, 16 a thread
  int cnt[NBIN / 1024], sum = 0;
#pragma unroll
  for (int i = 0; i < NBIN / 1024; i++) sum += cnt[i] = hist[NBIN - 1 - (t * (NBIN / 1024) + i)];
  int run = sum;
  for (int o = 1; o < 32; o <<= 1) {
    const int v = __shfl_up_sync(0xffffffffu, run, o);
    if (lane >= o) run += v;
  }
  if (lane == 31) ws[w] = run;
  if (t == 0) kb = NBIN;
  __syncthreads();
  int before = run - sum;
  for (int i = 0; i < w; i++) before += ws[i];
#pragma unroll
  for (int i = 0; i < NBIN / 1024; i++) {
    before += cnt[i];
    if (before <= MS) atomicMin(&kb, NBIN - 1 - (t * (NBIN / 1024) + i));
  }
  __syncthreads();
  const int key = max(kb, 1);
  if (t == 0) edge[0] = key;
  const double top = selv[0];
  int base = 0;
  for (int c0 = 0; c0 < n; c0 += 1024) {
    const int c = c0 + t;
    const bool in = c < n && bin_of(d[c], top) >= key;
    const unsigned m = __ballot_sync(0xffffffffu, in);
    __syncthreads();
    if (lane == 0) ws[w] = __popc(m);
    __syncthreads();
    int off = base, all = 0;
    for (int i = 0; i < 32; i++) {
      if (i < w) off += ws[i];
      all += ws[i];
    }
    if (in) idx[off + __popc(m & ((1u << lane) - 1))] = c;
    base += all;
  }
  for (int i = base + t; i < MS; i += 1024) idx[i] = -1;
  if (t == 0) edge[1] = base;
}

// Us[i][f] = U[f][idx[i]] (0 past the set); conj negates the imaginary part.
__global__ void __launch_bounds__(PT) gather_u(const double2* __restrict__ U, int nfunc, long ncand,
                                               const int* __restrict__ idx, int n, bool conj,
                                               double2* __restrict__ Us) {
  const long i = (long)blockIdx.x * PT + threadIdx.x;
  if (i >= (long)n * nfunc) return;
  const int p = idx[i / nfunc];
  double2 u = p >= 0 ? U[(i % nfunc) * ncand + p] : make_double2(0.0, 0.0);
  if (conj) u.y = -u.y;
  Us[i] = u;
}

// Ls[s][i] = L[s][idx[i]] (0 past the set), s < rows, rows ld apart.
__global__ void __launch_bounds__(PT) gather_l(const double* __restrict__ L, long ncand, const int* __restrict__ idx,
                                               int n, int ld, int rows, double* __restrict__ Ls) {
  const long i = (long)blockIdx.x * PT + threadIdx.x;
  if (i >= (long)rows * n) return;
  const int p = idx[i % n];
  Ls[(i / n) * ld + i % n] = p >= 0 ? L[(i / n) * ncand + p] : 0.0;
}

__global__ void __launch_bounds__(PT) abs2(const double2* __restrict__ B, long n, double* __restrict__ R) {
  const long i = (long)blockIdx.x * PT + threadIdx.x;
  if (i < n) R[i] = B[i].x * B[i].x + B[i].y * B[i].y;
}

// What a block of pivots leaves: their count, candidates, residuals at their
// selection, and W[s][t] = row s of the block at pivot t.
struct Picked {
  int count, pad;
  int piv[TP];
  double dp[TP];
  double trace[TP];     // sum of d after each pivot (finish_kernel)
  double W[TP][TP];
};

// Pivots from the set, one candidate per thread.  G: residual matrix on the
// set, lb: scratch of TP x MS.
__global__ void __launch_bounds__(1024) pivots_kernel(const double* __restrict__ G, const int* __restrict__ idx,
                                                      const double* __restrict__ d, const double* __restrict__ selv,
                                                      const int* __restrict__ edge, int most, double* __restrict__ lb,
                                                      Picked* __restrict__ out) {
  __shared__ double sv[32];
  __shared__ int si[32];
  const int c = threadIdx.x, lane = c & 31, w = c >> 5;
  const bool in = c < MS && idx[c] >= 0;
  double dc = in ? d[idx[c]] : -1.0;
  const double top = selv[0];
  int t = 0;
  for (; t < most; t++) {
    Best b{dc, c};       // positions are in ascending candidate order: ties go to the lowest
    for (int o = 16; o > 0; o >>= 1)
      b = better(b, Best{__shfl_xor_sync(0xffffffffu, b.v, o), __shfl_xor_sync(0xffffffffu, b.i, o)});
    __syncthreads();
    if (lane == 0) {
      sv[w] = b.v;
      si[w] = b.i;
    }
    __syncthreads();
    b = Best{sv[lane], si[lane]};
    for (int o = 16; o > 0; o >>= 1)
      b = better(b, Best{__shfl_xor_sync(0xffffffffu, b.v, o), __shfl_xor_sync(0xffffffffu, b.i, o)});
    if (!(b.v > 0.0) || bin_of(b.v, top) < edge[0]) break;
    const int p = b.i;
    if (c < MS) {
      double a = G[(long)p * MS + c];
      for (int s = 0; s < t; s++) a = fma(-lb[s * MS + c], lb[s * MS + p], a);
      const double l = a / sqrt(b.v);
      lb[t * MS + c] = l;
      if (in) dc = c == p ? 0.0 : fmax(dc - l * l, 0.0);
    }
    if (c < t) out->W[c][t] = lb[c * MS + p];
    if (c == 0) {
      out->piv[t] = idx[p];
      out->dp[t] = b.v;
    }
    __syncthreads();     // row t of lb before the next pivot reads it
  }
  if (c == 0) out->count = t;
}

// The block's rows of L for every candidate: R[t][c] holds |B|^2 minus the
// earlier rows' products; also d after the block and per-block sums of d after
// every pivot.  din may equal dout.
__global__ void __launch_bounds__(FT) finish_kernel(const double* __restrict__ R, int ncand, int T,
                                                    const Picked* __restrict__ pk, double* __restrict__ L,
                                                    const double* __restrict__ din, double* __restrict__ dout,
                                                    double* __restrict__ part) {
  __shared__ double sw[TP][TP], ss[FT / 32];
  __shared__ double sq[TP];
  __shared__ int sp[TP];
  for (int i = threadIdx.x; i < TP * TP; i += FT) sw[i / TP][i % TP] = pk->W[i / TP][i % TP];
  if (threadIdx.x < TP) {
    sq[threadIdx.x] = threadIdx.x < T ? sqrt(pk->dp[threadIdx.x]) : 1.0;
    sp[threadIdx.x] = threadIdx.x < T ? pk->piv[threadIdx.x] : -1;
  }
  __syncthreads();
  const int c = blockIdx.x * FT + threadIdx.x, lane = threadIdx.x & 31;
  const bool in = c < ncand;
  double d = in ? din[c] : 0.0, l[TP];
#pragma unroll
  for (int t = 0; t < TP; t++) {
    if (t < T) {
      double a = in ? R[(long)t * ncand + c] : 0.0;
#pragma unroll
      for (int s = 0; s < t; s++) a = fma(-l[s], sw[s][t], a);
      l[t] = a / sq[t];
      if (in) {
        L[(long)t * ncand + c] = l[t];
        d = c == sp[t] ? 0.0 : fmax(d - l[t] * l[t], 0.0);
      }
      double v = d;
      for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
      if (lane == 0) ss[threadIdx.x >> 5] = v;
      __syncthreads();
      if (threadIdx.x == 0) {
        v = 0.0;
        for (int i = 0; i < FT / 32; i++) v += ss[i];
        part[(long)t * gridDim.x + blockIdx.x] = v;
      }
      __syncthreads();
    } else {
      l[t] = 0.0;
    }
  }
  if (in) dout[c] = d;
}

// trace[t] = the sum of part[t][0 .. nb).  One block per pivot.
__global__ void __launch_bounds__(PT) trace_kernel(const double* __restrict__ part, int nb, Picked* __restrict__ pk) {
  __shared__ double ss[PT];
  double v = 0.0;
  for (int i = threadIdx.x; i < nb; i += PT) v += part[(long)blockIdx.x * nb + i];
  ss[threadIdx.x] = v;
  __syncthreads();
  for (int o = PT / 2; o > 0; o >>= 1) {
    if (threadIdx.x < o) ss[threadIdx.x] += ss[threadIdx.x + o];
    __syncthreads();
  }
  if (threadIdx.x == 0) pk->trace[blockIdx.x] = ss[0];
}

unsigned nblk(long n, int t) { return (unsigned)((n + t - 1) / t); }

// Device memory of the block form; any failure leaves it unused.
struct Blocks {
  int *idx = nullptr, *edge = nullptr, *hist = nullptr;
  double2 *Us = nullptr, *G2 = nullptr, *Up = nullptr, *Bc = nullptr;
  double *G = nullptr, *Ls = nullptr, *lb = nullptr, *R = nullptr, *part = nullptr, *dold = nullptr;
  Picked *pk = nullptr, *host = nullptr;
  void* lanes = nullptr;
  OzWork w;
  cudaError_t make(int nfunc, int ncand, int npts, cudaStream_t s) {
    cudaError_t e = cudaSuccess;
    auto get = [&](auto*& p, size_t n) {
      if (e == cudaSuccess) e = cudaMalloc((void**)&p, n * sizeof(*p));
    };
    get(idx, MS);
    get(edge, 2);
    get(hist, NBIN);
    get(Us, (size_t)MS * nfunc);
    get(G2, (size_t)MS * MS);
    get(G, (size_t)MS * MS);
    get(Ls, (size_t)npts * MS);
    get(lb, (size_t)TP * MS);
    get(Up, (size_t)TP * nfunc);
    get(Bc, (size_t)TP * ncand);
    get(R, (size_t)TP * ncand);
    get(part, (size_t)TP * nblk(ncand, FT));
    get(dold, ncand);
    get(pk, 1);
    if (e == cudaSuccess) e = cudaMalloc(&lanes, oz_lane_bytes(ncand, nfunc));
    if (e == cudaSuccess) e = cudaMallocHost((void**)&host, sizeof(Picked));
    const size_t least = std::max({oz_work_bytes(MS, MS, nfunc, 1), oz_work_min(npts), oz_lanes_work(TP, nfunc)});
    if (e == cudaSuccess)
      e = oz_alloc(w, std::max(least, std::min(oz_work_bytes(TP, ncand, (npts + 1) / 2, 1), (size_t)1 << 30)), least, s);
    if (e == cudaSuccess && !(oz_fits(MS, MS, nfunc, 1, false, w) && oz_fits(MS, MS, npts, 1, true, w) &&
                              oz_lanes_fit(TP, nfunc, w) && oz_fits(TP, ncand, npts, 1, true, w)))
      e = cudaErrorMemoryAllocation;
    return e;
  }
  void drop() {
    void* p[] = {idx, edge, hist, Us, G2, G, Ls, lb, Up, Bc, R, part, dold, pk, lanes};
    for (void* q : p)
      if (q) cudaFree(q);
    if (host) cudaFreeHost(host);
    oz_free(w);
    *this = Blocks{};
  }
};

}  // namespace

extern "C" thc_status thc_select_points(const double* U, int nfunc, int ncand, int npts, double rel_tol,
                                        int* points_host, int* npoints_host, double* resid_diag, void* stream) {
  if (!U || !points_host || !npoints_host || nfunc < 1 || ncand < 1 || npts < 1 || npts > ncand || rel_tol < 0)
    return THC_ERR_ARG;
  if ((uintptr_t)U & 15) return THC_ERR_ARG;
  cudaStream_t s = (cudaStream_t)stream;
  const int nb = (int)std::min<long>((ncand + PT - 1) / PT, 1024);
  double *d = nullptr, *L = nullptr, *pv = nullptr, *ps = nullptr, *selv = nullptr, *host = nullptr;
  int *pi = nullptr, *sel = nullptr;
  Blocks bk;
  thc_status st = THC_OK;
  cudaError_t e = cudaSuccess;
  auto fail = [&](cudaError_t err) {
    set_global_error(std::string("thc_select_points: ") + cudaGetErrorString(err));
    return err == cudaErrorMemoryAllocation ? THC_ERR_OOM : THC_ERR_CUDA;
  };
  do {
    if ((e = cudaMalloc(&d, sizeof(double) * ncand)) != cudaSuccess) break;
    if ((e = cudaMalloc(&L, sizeof(double) * (size_t)npts * ncand)) != cudaSuccess) break;
    if ((e = cudaMalloc(&pv, sizeof(double) * nb)) != cudaSuccess) break;
    if ((e = cudaMalloc(&ps, sizeof(double) * nb)) != cudaSuccess) break;
    if ((e = cudaMalloc(&pi, sizeof(int) * nb)) != cudaSuccess) break;
    if ((e = cudaMalloc(&sel, sizeof(int) * 4)) != cudaSuccess) break;
    if ((e = cudaMalloc(&selv, sizeof(double) * 2)) != cudaSuccess) break;
    if ((e = cudaMallocHost(&host, sizeof(double) * 4)) != cudaSuccess) break;
    const double2* u = (const double2*)U;
    const unsigned g = (unsigned)((ncand + PT - 1) / PT);
    // blocks of pivots where a block's products are worth their launches (about
    // 0.5 ms a block at the least, against 25 us and nfunc ncand / 1.3e11 s a
    // pivot) and there is room for their scratch
    bool blocks = npts >= TP / 2 && ncand >= 2 * MS && (double)nfunc * ncand >= 1e6 && 2L * nfunc <= OZ_MAX_K &&
                  npts <= OZ_MAX_K;
    if (blocks && bk.make(nfunc, ncand, npts, s) != cudaSuccess) {
      cudaGetLastError();
      bk.drop();
      blocks = false;
    }
    diag_kernel<<<g, PT, 0, s>>>(u, nfunc, ncand, d);
    if (blocks && (e = oz_lane_prepare(u, ncand, ncand, nfunc, bk.lanes, s)) != cudaSuccess) break;
    double tr0 = -1.0;
    int count = 0;
    // the pivots of one block, from a set that is not empty
    auto block = [&](int j) -> int {
      gather_u<<<nblk((long)MS * nfunc, PT), PT, 0, s>>>(u, nfunc, ncand, bk.idx, MS, false, bk.Us);
      if ((e = oz_gemm_z(A_MK_CONJ, B_NK, MS, MS, nfunc, bk.Us, nfunc, 0, bk.Us, nfunc, 0, bk.G2, MS, 0, 1, false, bk.w, s)) !=
          cudaSuccess)
        return 0;
      abs2<<<nblk((long)MS * MS, PT), PT, 0, s>>>(bk.G2, (long)MS * MS, bk.G);
      if (j > 0) {
        gather_l<<<nblk((long)j * MS, PT), PT, 0, s>>>(L, ncand, bk.idx, MS, MS, j, bk.Ls);
        if ((e = oz_gemm_d(true, true, MS, MS, j, bk.Ls, MS, bk.Ls, MS, bk.G, MS, -1.0, true, false, bk.w, s)) != cudaSuccess)
          return 0;
      }
      pivots_kernel<<<1, 1024, 0, s>>>(bk.G, bk.idx, d, selv, bk.edge, std::min(TP, npts - j), bk.lb, bk.pk);
      if ((e = cudaMemcpyAsync(bk.host, bk.pk, offsetof(Picked, dp), cudaMemcpyDeviceToHost, s)) != cudaSuccess) return 0;
      if ((e = cudaStreamSynchronize(s)) != cudaSuccess) return 0;
      const int T = bk.host->count;
      if (T == 0) return 0;
      gather_u<<<nblk((long)T * nfunc, PT), PT, 0, s>>>(u, nfunc, ncand, bk.pk->piv, T, true, bk.Up);
      if ((e = oz_gemm_z_lanes(A_MK, T, ncand, nfunc, bk.Up, nfunc, bk.lanes, bk.Bc, ncand, bk.w, s)) != cudaSuccess)
        return 0;
      abs2<<<nblk((long)T * ncand, PT), PT, 0, s>>>(bk.Bc, (long)T * ncand, bk.R);
      if (j > 0) {
        gather_l<<<nblk((long)j * T, PT), PT, 0, s>>>(L, ncand, bk.pk->piv, T, TP, j, bk.Ls);
        if ((e = oz_gemm_d(true, true, T, ncand, j, bk.Ls, TP, L, ncand, bk.R, ncand, -1.0, true, false, bk.w,
                           s)) != cudaSuccess)
          return 0;
      }
      if ((e = cudaMemcpyAsync(bk.dold, d, sizeof(double) * ncand, cudaMemcpyDeviceToDevice, s)) != cudaSuccess) return 0;
      const unsigned fb = nblk(ncand, FT);
      finish_kernel<<<fb, FT, 0, s>>>(bk.R, ncand, T, bk.pk, L + (long)j * ncand, bk.dold, d, bk.part);
      trace_kernel<<<T, PT, 0, s>>>(bk.part, (int)fb, bk.pk);
      if ((e = cudaMemcpyAsync(bk.host->trace, bk.pk->trace, sizeof(double) * TP, cudaMemcpyDeviceToHost, s)) != cudaSuccess)
        return 0;
      if ((e = cudaStreamSynchronize(s)) != cudaSuccess) return 0;
      // the selection ends where the trace falls to rel_tol of the start's, also inside a block
      for (int t = 0; t + 1 < T; t++)
        if (!(bk.host->trace[t] > rel_tol * tr0)) {
          finish_kernel<<<fb, FT, 0, s>>>(bk.R, ncand, t + 1, bk.pk, L + (long)j * ncand, bk.dold, d, bk.part);
          e = cudaGetLastError();
          return t + 1;
        }
      return T;
    };
    // single pivots to take before the next block, and after the next one that does not pay: one of fewer pivots
    // than its 0.5 ms of launches take one by one (17 at nfunc ncand = 1e6, 2 at 1e8)
    int skip = 0, back = 8;
    const int pays = 2 + (int)(0.5e-3 / (25e-6 + (double)nfunc * ncand / 1.3e11));
    for (int j = 0; j < npts;) {
      argmax_partial<<<nb, PT, 0, s>>>(d, ncand, pv, pi, ps);
      argmax_final<<<1, PT, 0, s>>>(pv, pi, ps, nb, sel, selv);
      const bool try_block = blocks && skip == 0;
      if (try_block) {
        if ((e = cudaMemsetAsync(bk.hist, 0, sizeof(int) * NBIN, s)) != cudaSuccess) break;
        hist_kernel<<<nb, PT, 0, s>>>(d, ncand, selv, bk.hist);
        pick_kernel<<<1, 1024, 0, s>>>(d, ncand, selv, bk.hist, bk.idx, bk.edge);
        if ((e = cudaMemcpyAsync((int*)(host + 3), bk.edge + 1, sizeof(int), cudaMemcpyDeviceToHost, s)) != cudaSuccess)
          break;
      }
      if ((e = cudaMemcpyAsync(host, selv, 2 * sizeof(double), cudaMemcpyDeviceToHost, s)) != cudaSuccess) break;
      if ((e = cudaMemcpyAsync((int*)(host + 2), sel, sizeof(int), cudaMemcpyDeviceToHost, s)) != cudaSuccess)
        break;
      if ((e = cudaStreamSynchronize(s)) != cudaSuccess) break;
      const double trace = host[1];
      if (j == 0) tr0 = trace;
      if (!(trace > rel_tol * tr0) || !(host[0] > 0.0)) break;   // rank reached
      if (skip > 0) skip--;
      if (try_block) {
        const int T = *(int*)(host + 3) > 0 ? block(j) : 0;
        if (e != cudaSuccess) break;
        if (T < pays && j + T < npts) {
          skip = back;
          back = std::min(2 * back, 1024);
        } else {
          back = 8;
        }
        if (T > 0) {
          for (int t = 0; t < T; t++) points_host[j + t] = bk.host->piv[t];
          j += T;
          count = j;
          continue;
        }
      }
      points_host[j] = *(int*)(host + 2);
      column_kernel<<<(unsigned)((ncand + 31) / 32), 32 * CW, 0, s>>>(u, nfunc, ncand, j, sel, selv, L, d);
      if ((e = cudaGetLastError()) != cudaSuccess) break;
      count = ++j;
    }
    if (e == cudaSuccess && blocks) {
      int h = 0;
      e = cudaMemcpyAsync(&h, bk.w.err, sizeof(int), cudaMemcpyDeviceToHost, s);
      if (e == cudaSuccess) e = cudaStreamSynchronize(s);
      if (h) {
        set_global_error("thc_select_points: a device wait of a tensor-core product timed out");
        st = THC_ERR_TIMEOUT;
        break;
      }
    }
    if (e != cudaSuccess) break;
    for (int j = count; j < npts; j++) points_host[j] = -1;
    *npoints_host = count;
    if (resid_diag &&
        (e = cudaMemcpyAsync(resid_diag, d, sizeof(double) * ncand, cudaMemcpyDeviceToDevice, s)) != cudaSuccess)
      break;
    e = cudaStreamSynchronize(s);
  } while (0);
  if (e != cudaSuccess) st = fail(e);
  if (d) cudaFree(d);
  if (L) cudaFree(L);
  if (pv) cudaFree(pv);
  if (ps) cudaFree(ps);
  if (pi) cudaFree(pi);
  if (sel) cudaFree(sel);
  if (selv) cudaFree(selv);
  if (host) cudaFreeHost(host);
  bk.drop();
  return st;
}
