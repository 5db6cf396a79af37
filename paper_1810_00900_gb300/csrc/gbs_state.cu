// State construction and Sigma^-1 click blocks.
//
//  - state_params_kernel / build_V_kernel: the covariance of squeezed vacuum
//    followed by an interferometer and loss (paper Sec. II, Eq. 1; inputs as in
//    Sec. III; loss as in Sec. IV):
//        V = S S^+ / 2,  S = [[U ch R, U sh R], [U* sh R, U* ch R]]
//    blockwise A = U diag(cosh 2r) U^+ / 2, B = U diag(sinh 2r) U^T / 2,
//    V = [[A, B], [B*, A*]], then V <- eta V + (1 - eta) I/2.
//  - Closed-form inverse: with E = blockdiag(U, U*) P, P mixing (a_l, a_l^+)
//    into (1, +-1)/sqrt2, Sigma = V + I/2 = E diag(d+, d-) E^+ with
//    d+- = (eta e^{+-2r} + 2 - eta)/2, hence
//        (Sigma^-1)_{a_j a_k}   = sum_l U_jl conj(U_kl) alpha_l
//        (Sigma^-1)_{a_j a^+_k} = sum_l U_jl U_kl beta_l
//    with alpha = (1/d+ + 1/d-)/2, beta = (1/d+ - 1/d-)/2, and
//    log det Sigma = sum_l log(d+ d-).  O(N^2 M) per click block.
//  - States given only by V: Sigma is inverted by the sweep operator in blocks of 16
//    pivots (no pivoting; Sigma is Hermitian positive definite), on its lower triangle;
//    log det Sigma is the sum of the logs of the pivots.
#include <algorithm>
#include <cmath>
#include <cstring>
#include <vector>

#include "gbs_internal.h"
#include "gbs_num.cuh"

namespace gbs {

// packed lower-triangle index of entry (a, b), a >= b
static __host__ __device__ constexpr int tri(int a, int b) { return a * (a + 1) / 2 + b; }

__global__ void state_params_kernel(const double* __restrict__ r, double eta, int M, double* __restrict__ alpha,
                                    double* __restrict__ beta, double* __restrict__ ch2, double* __restrict__ sh2,
                                    double* __restrict__ logd) {
  const int l = blockIdx.x * blockDim.x + threadIdx.x;
  if (l >= M) return;
  const double e = exp(2.0 * r[l]);
  const double dp = 0.5 * (eta * e + 2.0 - eta);
  const double dm = 0.5 * (eta / e + 2.0 - eta);
  alpha[l] = 0.5 * (1.0 / dp + 1.0 / dm);
  beta[l] = 0.5 * (1.0 / dp - 1.0 / dm);
  ch2[l] = 0.5 * cosh(2.0 * r[l]);
  sh2[l] = 0.5 * sinh(2.0 * r[l]);
  logd[l] = log(dp) + log(dm);
}

// Fixed-order double-double sum of x[0..n), or of the logarithms (LOG), by one block.
template <bool LOG>
__global__ void sum_dd_kernel(const double* __restrict__ x, int n, double* __restrict__ out) {
  // strided per-thread sums, then a fixed-order shuffle tree within each warp
  // and across the (at most 32) warps: deterministic, and no serial loop
  dd acc = dd_make(0.0);
  for (int i = threadIdx.x; i < n; i += blockDim.x) acc = acc + (LOG ? log(x[i]) : x[i]);
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
  for (int off = 16; off > 0; off >>= 1)
    acc = acc + dd{__shfl_down_sync(0xffffffffu, acc.hi, off), __shfl_down_sync(0xffffffffu, acc.lo, off)};
  __shared__ dd sh[32];
  if (lane == 0) sh[warp] = acc;
  __syncthreads();
  if (warp == 0) {
    const int nw = (blockDim.x + 31) >> 5;
    dd t = lane < nw ? sh[lane] : dd_make(0.0);
#pragma unroll
    for (int off = 16; off > 0; off >>= 1)
      t = t + dd{__shfl_down_sync(0xffffffffu, t.hi, off), __shfl_down_sync(0xffffffffu, t.lo, off)};
    if (lane == 0) out[0] = t.hi + t.lo;
  }
}

// V from the factors, an 8 x 8 tile of mode pairs (j, k), j >= k, per CTA of 64 threads;
// the other half by symmetry (A Hermitian, B symmetric).  Bound by the FP64 pipe: 8 FMAs
// per (pair, l), with the rows of U weighted by cosh and sinh once per tile as they are
// staged (a thread per pair of the full square with the weights applied to each product
// took 16 operations per (j, k, l), and read U's rows a thread apart).  Small tiles, so
// that the triangle's CTAs fill the SMs evenly.  The sums go in runs of kVL, whose rounding
// is below that of one chain (M = 333, relative to a wider sum: 5.2e-16, 8.9e-16 with one).  M = 333: 648 -> 290 us, of which 243
// are the FMAs.
constexpr int kVT = 8, kVL = 32;
__global__ void __launch_bounds__(64) build_V_kernel(const cplx<double>* __restrict__ U, const double* __restrict__ ch2,
                                                     const double* __restrict__ sh2, double eta, int M,
                                                     cplx<double>* __restrict__ V) {
  __shared__ cplx<double> sc[kVT][kVL + 1], ss[kVT][kVL + 1], sy[kVT][kVL + 1];
  int tj = (int)((sqrtf(8.0f * (float)blockIdx.x + 1.0f) - 1.0f) * 0.5f);
  while (tj * (tj + 1) / 2 > (int)blockIdx.x) --tj;
  while ((tj + 1) * (tj + 2) / 2 <= (int)blockIdx.x) ++tj;
  const int tk = (int)blockIdx.x - tj * (tj + 1) / 2;
  const int lj = threadIdx.x / kVT, lk = threadIdx.x % kVT;
  const int j = tj * kVT + lj, k = tk * kVT + lk;
  double ar = 0, ai = 0, br = 0, bi = 0;
  for (int l0 = 0; l0 < M; l0 += kVL) {
    for (int e = threadIdx.x; e < kVT * kVL; e += 64) {
      const int r = e / kVL, c = e % kVL, l = l0 + c;
      const bool okl = l < M;
      const int rj = tj * kVT + r, rk = tk * kVT + r;
      const cplx<double> x = okl && rj < M ? U[(long long)rj * M + l] : cplx<double>{0, 0};
      const double wc = okl ? ch2[l] : 0.0, ws = okl ? sh2[l] : 0.0;
      sc[r][c] = {x.re * wc, x.im * wc};
      ss[r][c] = {x.re * ws, x.im * ws};
      sy[r][c] = okl && rk < M ? U[(long long)rk * M + l] : cplx<double>{0, 0};
    }
    __syncthreads();
    double car = 0, cai = 0, cbr = 0, cbi = 0;  // this run's sums
    const int len = min(kVL, M - l0);  // (all of a run for M = 2 as well took 8 us more)
#pragma unroll 4
    for (int c = 0; c < len; ++c) {
      const cplx<double> y = sy[lk][c], p = sc[lj][c], q = ss[lj][c];
      // x conj(y) cosh(2r)/2 and x y sinh(2r)/2
      car = fma(p.re, y.re, fma(p.im, y.im, car));
      cai = fma(p.im, y.re, fma(-p.re, y.im, cai));
      cbr = fma(q.re, y.re, fma(-q.im, y.im, cbr));
      cbi = fma(q.re, y.im, fma(q.im, y.re, cbi));
    }
    ar += car;
    ai += cai;
    br += cbr;
    bi += cbi;
    __syncthreads();
  }
  if (j >= M || k > j) return;
  const double diag = (j == k) ? 0.5 * (1.0 - eta) : 0.0;
  const long long D = 2LL * M;
  const cplx<double> A{eta * ar + diag, j == k ? 0.0 : eta * ai}, Ac{A.re, -A.im}, B{eta * br, eta * bi}, Bc{B.re, -B.im};
  V[(long long)j * D + k] = A;
  V[(long long)k * D + j] = Ac;
  V[(long long)j * D + k + M] = B;
  V[(long long)k * D + j + M] = B;
  V[(long long)(j + M) * D + k] = Bc;
  V[(long long)(k + M) * D + j] = Bc;
  V[(long long)(j + M) * D + k + M] = Ac;
  V[(long long)(k + M) * D + j + M] = A;
}

// Click block from the factors: one warp per mode pair (j >= k).  Output packed
// lower triangle of the 2N x 2N matrix (entry (a, b), a >= b, at tri(a, b)).
__global__ void sigma_inv_block_kernel(const cplx<double>* __restrict__ U, const double* __restrict__ alpha,
                                       const double* __restrict__ beta, int M, ModeList S, int N, int real_basis,
                                       void* __restrict__ out) {
  const int warp = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const int lane = threadIdx.x & 31;
  const int npairs = N * (N + 1) / 2;
  if (warp >= npairs) return;
  int j = 0;
  while ((j + 1) * (j + 2) / 2 <= warp) ++j;
  const int k = warp - j * (j + 1) / 2;
  const cplx<double>* uj = U + (long long)S.m[j] * M;
  const cplx<double>* uk = U + (long long)S.m[k] * M;
  double ar = 0, ai = 0, br = 0, bi = 0;
  for (int l = lane; l < M; l += 32) {
    const cplx<double> x = uj[l], y = uk[l];
    const double pr = x.re * y.re + x.im * y.im, pi = x.im * y.re - x.re * y.im;
    const double qr = x.re * y.re - x.im * y.im, qi = x.re * y.im + x.im * y.re;
    ar = fma(pr, alpha[l], ar);
    ai = fma(pi, alpha[l], ai);
    br = fma(qr, beta[l], br);
    bi = fma(qi, beta[l], bi);
  }
#pragma unroll
  for (int off = 16; off > 0; off >>= 1) {
    ar += __shfl_down_sync(0xffffffffu, ar, off);
    ai += __shfl_down_sync(0xffffffffu, ai, off);
    br += __shfl_down_sync(0xffffffffu, br, off);
    bi += __shfl_down_sync(0xffffffffu, bi, off);
  }
  if (lane != 0) return;
  if (j == k) ai = 0.0;  // A is Hermitian: real diagonal
  const int a0 = 2 * j, b0 = 2 * k;
  if (real_basis) {
    double* o = (double*)out;
    // q^+ [[A, B], [B*, A*]] q with q = [[1, i], [1, -i]]/sqrt2 (columns x, p)
    o[tri(a0, b0)] = ar + br;
    o[tri(a0 + 1, b0)] = ai + bi;
    o[tri(a0 + 1, b0 + 1)] = ar - br;
    if (j != k) o[tri(a0, b0 + 1)] = bi - ai;
  } else {
    cplx<double>* o = (cplx<double>*)out;
    o[tri(a0, b0)] = {ar, ai};
    o[tri(a0 + 1, b0)] = {br, -bi};
    o[tri(a0 + 1, b0 + 1)] = {ar, -ai};
    if (j != k) o[tri(a0, b0 + 1)] = {br, bi};
  }
}

// Click block from a dense Sigma^-1 (block order): one thread per mode pair.
__global__ void gather_inv_block_kernel(const cplx<double>* __restrict__ Si, int M, ModeList S, int N,
                                        int real_basis, void* __restrict__ out) {
  const int p = blockIdx.x * blockDim.x + threadIdx.x;
  if (p >= N * (N + 1) / 2) return;
  int j = 0;
  while ((j + 1) * (j + 2) / 2 <= p) ++j;
  const int k = p - j * (j + 1) / 2;
  const long long D = 2LL * M;
  const int rj = S.m[j], rk = S.m[k];
  cplx<double> h00 = Si[rj * D + rk], h01 = Si[rj * D + rk + M];
  cplx<double> h10 = Si[(rj + M) * D + rk], h11 = Si[(rj + M) * D + rk + M];
  const int a0 = 2 * j, b0 = 2 * k;
  if (real_basis) {
    double* o = (double*)out;
    o[tri(a0, b0)] = 0.5 * (h00.re + h01.re + h10.re + h11.re);
    o[tri(a0 + 1, b0)] = 0.5 * ((h00.im + h01.im) - (h10.im + h11.im));
    o[tri(a0 + 1, b0 + 1)] = 0.5 * ((h00.re - h01.re) - (h10.re - h11.re));
    if (j != k) o[tri(a0, b0 + 1)] = -0.5 * (h00.im - h01.im + h10.im - h11.im);
  } else {
    cplx<double>* o = (cplx<double>*)out;
    if (j == k) { h00.im = 0.0; h11.im = 0.0; }
    o[tri(a0, b0)] = h00;
    o[tri(a0 + 1, b0)] = h10;
    o[tri(a0 + 1, b0 + 1)] = h11;
    if (j != k) o[tri(a0, b0 + 1)] = h01;
  }
}

// Sigma = V + I/2; flags non-finite entries and sums each row's magnitudes (a warp per
// row; Gershgorin's bound on the largest eigenvalue).
__global__ void sigma_from_V_kernel(const cplx<double>* __restrict__ V, int D, cplx<double>* __restrict__ X,
                                    double* __restrict__ rowsum, int* __restrict__ bad) {
  const int i = (int)((blockIdx.x * blockDim.x + threadIdx.x) >> 5), lane = threadIdx.x & 31;
  if (i >= D) return;
  double sum = 0.0;
  bool fin = true;
  for (int j = lane; j < D; j += 32) {
    cplx<double> v = V[(long long)i * D + j];
    fin &= isfinite(v.re) && isfinite(v.im);
    sum += hypot(v.re, v.im);
    if (i == j) v.re += 0.5;
    X[(long long)i * D + j] = v;
  }
#pragma unroll
  for (int off = 16; off > 0; off >>= 1) sum += __shfl_down_sync(0xffffffffu, sum, off);
  if (!fin) atomicExch(bad, 1);
  if (lane == 0) rowsum[i] = sum + 0.5;
}

// Inverse of Sigma by the sweep operator in blocks of kSW pivots, on the lower triangle,
// in place.  Sweeping pivot block K (P = X[K, K], C = X[:, K], G = C P^-1):
//   X[I, J] -= C[I] G[J]^+,  X[I, K] = G[I],  X[K, K] = -P^-1,
// which keeps X Hermitian; after all blocks X = -Sigma^-1.  The pivots on the way are
// those of one-by-one elimination.  Two launches per block: the panel (C and G), and the
// update, in which one extra CTA forms and inverts the next pivot block meanwhile -- the
// chain of scalar pivots is what bounds the whole (0.5 us each), then the FP64 pipe.
// One launch per scalar pivot over the full matrix took 5.2 us a pivot: D = 240 1.27 ms,
// now 0.37.
constexpr int kSW = 16;

// 1/x of a positive double: two Newton steps from the single-precision reciprocal of
// its significand (1 FP64 division is a chain of ten FP64 operations).
__device__ __forceinline__ double recip_pos(double x) {
  const long long b = __double_as_longlong(x);
  const int e = (int)(b >> 52) & 0x7ff;
  if (e == 0 || e >= 2040) return 1.0 / x;  // subnormal, or a reciprocal that would be
  const double m = __longlong_as_double((b & 0xfffffffffffffll) | 0x3ff0000000000000ll);  // [1, 2)
  double y = (double)__frcp_rn((float)m);
  y = fma(y, fma(-m, y, 1.0), y);
  y = fma(y, fma(-m, y, 1.0), y);
  return y * __longlong_as_double((long long)(2046 - e) << 52);
}

// Inverts the b x b Hermitian block S (lower triangle, shared memory) in place by scalar
// sweeps; piv[t]: the scalar pivots.  All threads of the CTA (256) take part: one warp
// forms the pivot's reciprocal and column, a thread per entry of the triangle (packed, so
// that five warps' FP64 instructions and not eight share the pipe) the update.
__device__ __forceinline__ void invert_block(cplx<double> (*S)[kSW + 1], int b, double* __restrict__ piv,
                                             int* __restrict__ status) {
  __shared__ cplx<double> col[kSW], g[kSW];  // the pivot's column, and over the pivot
  __shared__ double s_ip;
  const int e = threadIdx.x;
  int i = (int)((sqrtf(8.0f * (float)e + 1.0f) - 1.0f) * 0.5f);
  while (i * (i + 1) / 2 > e) --i;
  while ((i + 1) * (i + 2) / 2 <= e) ++i;
  const int j = e - i * (i + 1) / 2;
  __syncthreads();
  for (int t = 0; t < b; ++t) {
    if (threadIdx.x < 32) {
      const int r = threadIdx.x;
      const double p = S[t][t].re, ip = recip_pos(p);
      if (r < b) {
        const cplx<double> c = r >= t ? S[r][t] : cplx<double>{S[t][r].re, -S[t][r].im};
        col[r] = c;
        g[r] = {c.re * ip, c.im * ip};
      }
      if (r == 0) {
        s_ip = ip;
        piv[t] = p;
        if (!(p > 0.0)) atomicExch(status, (int)3);
      }
    }
    __syncthreads();
    if (i < b) {
      cplx<double> y;
      if (i == t) {
        y = j == t ? cplx<double>{-s_ip, 0.0} : cplx<double>{g[j].re, -g[j].im};
      } else if (j == t) {
        y = g[i];
      } else {
        const cplx<double> c = col[i], h = g[j], x = S[i][j];  // x - c conj(h)
        y.re = fma(-c.re, h.re, fma(-c.im, h.im, x.re));
        y.im = i == j ? 0.0 : fma(-c.im, h.re, fma(c.re, h.im, x.im));
      }
      S[i][j] = y;
    }
    __syncthreads();
  }
  // sweeping left -S^-1
  if (i < b) S[i][j] = {-S[i][j].re, -S[i][j].im};
  __syncthreads();
}

// The first pivot block's inverse (Pinv: kSW x kSW, full); X is swept where that is all of it.
__global__ void __launch_bounds__(256) sweep_first_kernel(cplx<double>* __restrict__ X, int D,
                                                          cplx<double>* __restrict__ Pinv, double* __restrict__ piv,
                                                          int* __restrict__ status) {
  __shared__ cplx<double> S[kSW][kSW + 1];
  const int b = min(kSW, D), i = threadIdx.x / kSW, j = threadIdx.x % kSW;
  if (i < b && j <= i) S[i][j] = X[(long long)i * D + j];
  invert_block(S, b, piv, status);
  if (i >= b || j >= b) return;
  const cplx<double> p = j <= i ? S[i][j] : cplx<double>{S[j][i].re, -S[j][i].im};
  Pinv[i * kSW + j] = p;
  if (D <= kSW && j <= i) X[(long long)i * D + j] = {-p.re, -p.im};
}

// Panel of pivot block k0: C = X[:, K] and G = C P^-1 for 16 rows per CTA; and a copy
// (Xk) of the next pivot block for the update's extra CTA.
__global__ void __launch_bounds__(256) sweep_panel_kernel(const cplx<double>* __restrict__ X, int D, int k0,
                                                          const cplx<double>* __restrict__ Pinv,
                                                          cplx<double>* __restrict__ C, cplx<double>* __restrict__ G,
                                                          cplx<double>* __restrict__ Xk) {
  __shared__ cplx<double> c[kSW][kSW + 1], q[kSW][kSW + 1];
  const int b = min(kSW, D - k0), r = threadIdx.x / kSW, t = threadIdx.x % kSW;
  const int i = blockIdx.x * kSW + r;
  cplx<double> x{0, 0};
  if (i < D && t < b && (i < k0 || i >= k0 + b)) {
    if (i >= k0) {
      x = X[(long long)i * D + k0 + t];
    } else {
      x = X[(long long)(k0 + t) * D + i];
      x.im = -x.im;
    }
  }
  if ((int)blockIdx.x == k0 / kSW + 1 && i < D && t <= r) Xk[r * kSW + t] = X[(long long)i * D + i - r + t];
  c[r][t] = x;
  q[r][t] = r < b && t < b ? Pinv[r * kSW + t] : cplx<double>{0, 0};
  __syncthreads();
  double gr = 0, gi = 0;
#pragma unroll
  for (int u = 0; u < kSW; ++u) {
    const cplx<double> a = c[r][u], p = q[u][t];
    gr = fma(a.re, p.re, fma(-a.im, p.im, gr));
    gi = fma(a.re, p.im, fma(a.im, p.re, gi));
  }
  if (i < D) {
    C[(long long)i * kSW + t] = x;
    G[(long long)i * kSW + t] = {gr, gi};
  }
}

// Update of the lower triangle, 16 x 16 entries per CTA; the last CTA forms the next
// pivot block from C and G as well and inverts it.
__global__ void __launch_bounds__(256) sweep_update_kernel(cplx<double>* __restrict__ X, int D, int k0, int ntiles,
                                                           const cplx<double>* __restrict__ Pinv,
                                                           const cplx<double>* __restrict__ C,
                                                           const cplx<double>* __restrict__ G,
                                                           const cplx<double>* __restrict__ Xk,
                                                           cplx<double>* __restrict__ Pnext, double* __restrict__ piv,
                                                           int* __restrict__ status) {
  __shared__ cplx<double> c[kSW][kSW + 1], g[kSW][kSW + 1];
  const int r = threadIdx.x / kSW, t = threadIdx.x % kSW;
  const bool next = (int)blockIdx.x == ntiles;
  int ti, tj;
  if (next) {
    ti = tj = k0 / kSW + 1;  // the next pivot block is a diagonal tile
  } else {
    ti = (int)((sqrtf(8.0f * (float)blockIdx.x + 1.0f) - 1.0f) * 0.5f);
    while (ti * (ti + 1) / 2 > (int)blockIdx.x) --ti;
    while ((ti + 1) * (ti + 2) / 2 <= (int)blockIdx.x) ++ti;
    tj = (int)blockIdx.x - ti * (ti + 1) / 2;
  }
  const int i0 = ti * kSW, j0 = tj * kSW, i = i0 + r, j = j0 + t;
  c[r][t] = i < D ? C[(long long)i * kSW + t] : cplx<double>{0, 0};
  g[r][t] = j0 + r < D ? G[(long long)(j0 + r) * kSW + t] : cplx<double>{0, 0};
  __syncthreads();
  const bool in = i < D && j <= i;
  cplx<double> y{0, 0};
  if (ti == k0 / kSW && tj == ti) {
    if (in) {
      const cplx<double> p = Pinv[r * kSW + t];
      y = {-p.re, -p.im};
    }
  } else if (tj == k0 / kSW) {
    if (in) y = G[(long long)i * kSW + t];
  } else if (ti == k0 / kSW) {
    if (in) {
      y = g[t][r];
      y.im = -y.im;
    }
  } else {
    double xr = 0, xi = 0;
#pragma unroll
    for (int u = 0; u < kSW; ++u) {
      const cplx<double> a = c[r][u], h = g[t][u];  // a conj(h)
      xr = fma(a.re, h.re, fma(a.im, h.im, xr));
      xi = fma(a.im, h.re, fma(-a.re, h.im, xi));
    }
    if (in) {
      // the next block reads its entries from their copy: another CTA writes them here
      const cplx<double> x = next ? Xk[r * kSW + t] : X[(long long)i * D + j];
      y = {x.re - xr, i == j ? 0.0 : x.im - xi};
    }
  }
  if (!next) {
    if (in) X[(long long)i * D + j] = y;
    return;
  }
  __shared__ cplx<double> S[kSW][kSW + 1];
  if (in) S[r][t] = y;
  const int bn = min(kSW, D - i0);
  invert_block(S, bn, piv + i0, status);
  if (r < bn && t < bn) Pnext[r * kSW + t] = t <= r ? S[r][t] : cplx<double>{S[t][r].re, -S[t][r].im};
}

// Sigma^-1 = -X, both triangles.
__global__ void sweep_negate_kernel(const cplx<double>* __restrict__ X, int D, cplx<double>* __restrict__ Y) {
  const long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= (long long)D * D) return;
  const int i = (int)(t / D), j = (int)(t % D);
  if (j <= i) {
    const cplx<double> x = X[t];
    Y[t] = {-x.re, -x.im};
  } else {
    const cplx<double> x = X[(long long)j * D + i];
    Y[t] = {-x.re, x.im};
  }
}

// ------------------------------------------------------------ host side --

static gbs_status alloc_state(gbs_ctx* ctx, int M, gbs_state** out) {
  gbs_state* st = new gbs_state();
  st->ctx = ctx;
  st->M = M;
  *out = st;
  return GBS_OK;
}

// The covariance V of a factor-built state, on first use (sampling, V_out).
gbs_status ensure_V(gbs_ctx* ctx, gbs_state* st) {
  if (st->V.ptr) return GBS_OK;
  const int M = st->M;
  const size_t MM = (size_t)M * M;
  DevBuf tmp;
  gbs_status e;
  if ((e = dev_alloc(ctx, st->V, 4 * MM * 16)) || (e = dev_alloc(ctx, tmp, (3 * (size_t)M + 1) * 8))) {
    dev_free(ctx, tmp);
    return e;
  }
  double* ch2 = (double*)tmp.ptr;
  double* sh2 = ch2 + M;
  double* logd = sh2 + M;
  cudaStream_t s = ctx->stream;
  // alpha/beta are already in place: rewrite them with identical values
  state_params_kernel<<<(M + 127) / 128, 128, 0, s>>>((const double*)st->r.ptr, st->eta, M, (double*)st->alpha.ptr,
                                                      (double*)st->beta.ptr, ch2, sh2, logd);
  const unsigned vt = (unsigned)((M + kVT - 1) / kVT);
  build_V_kernel<<<vt * (vt + 1) / 2, kVT * kVT, 0, s>>>((const cplx<double>*)st->U.ptr, ch2, sh2, st->eta, M,
                                                                (cplx<double>*)st->V.ptr);
  count_launch(ctx, 2);
  if ((e = check_cuda(ctx, cudaGetLastError(), "build V")) ||
      (e = stream_sync(ctx))) {
    dev_free(ctx, tmp);
    return e;
  }
  dev_free(ctx, tmp);
  return GBS_OK;
}

gbs_status state_build(gbs_ctx* ctx, int M, const double* U, const double* r, double eta, double* V_out,
                       gbs_state** out) {
  if (M < 1 || !U || !r || !out) return set_error(ctx, GBS_EINVAL, "gbs_build_state: bad arguments");
  if (!(eta > 0.0 && eta <= 1.0)) return set_error(ctx, GBS_EINVAL, "gbs_build_state: eta must be in (0, 1]");
  for (int l = 0; l < M; ++l)
    if (!std::isfinite(r[l])) return set_error(ctx, GBS_EINVAL, "gbs_build_state: non-finite squeezing");
  for (long long i = 0; i < 2LL * M * M; ++i)
    if (!std::isfinite(U[i])) return set_error(ctx, GBS_EINVAL, "gbs_build_state: non-finite U");
  gbs_state* st = nullptr;
  alloc_state(ctx, M, &st);
  st->has_factors = true;
  st->eta = eta;
  // largest eigenvalue of Sigma: max over modes of d+ = (eta e^(2|r|) + 2 - eta) / 2
  for (int l = 0; l < M; ++l)
    st->sigma_max = std::max(st->sigma_max, 0.5 * (eta * std::exp(2.0 * std::fabs(r[l])) + 2.0 - eta));
  const size_t MM = (size_t)M * M;
  DevBuf tmp;
  gbs_status e;
  auto fail = [&](gbs_status code) {
    dev_free(ctx, tmp);
    gbs_state_free(st);
    return code;
  };
  if ((e = dev_alloc(ctx, st->U, MM * 16)) || (e = dev_alloc(ctx, st->r, M * 8)) ||
      (e = dev_alloc(ctx, st->alpha, M * 8)) || (e = dev_alloc(ctx, st->beta, M * 8)) ||
      (e = dev_alloc(ctx, tmp, (3 * (size_t)M + 1) * 8)))
    return fail(e);
  cudaStream_t s = ctx->stream;
  if ((e = check_cuda(ctx, cudaMemcpyAsync(st->U.ptr, U, MM * 16, cudaMemcpyHostToDevice, s), "copy U")) ||
      (e = check_cuda(ctx, cudaMemcpyAsync(st->r.ptr, r, M * 8, cudaMemcpyHostToDevice, s), "copy r")))
    return fail(e);
  double* ch2 = (double*)tmp.ptr;
  double* sh2 = ch2 + M;
  double* logd = sh2 + M;
  double* ld_out = logd + M;
  state_params_kernel<<<(M + 127) / 128, 128, 0, s>>>((const double*)st->r.ptr, eta, M, (double*)st->alpha.ptr,
                                                      (double*)st->beta.ptr, ch2, sh2, logd);
  sum_dd_kernel<false><<<1, 256, 0, s>>>(logd, M, ld_out);
  count_launch(ctx, 2);
  if ((e = check_cuda(ctx, cudaGetLastError(), "state kernels"))) return fail(e);
  if ((e = check_cuda(ctx, cudaMemcpyAsync(&st->logdet_sigma, ld_out, 8, cudaMemcpyDeviceToHost, s), "copy logdet")))
    return fail(e);
  if ((e = stream_sync(ctx))) return fail(e);
  dev_free(ctx, tmp);
  if (V_out) {
    if ((e = ensure_V(ctx, st))) return fail(e);
    if ((e = check_cuda(ctx, cudaMemcpyAsync(V_out, st->V.ptr, 4 * MM * 16, cudaMemcpyDeviceToHost, s), "copy V")) ||
        (e = stream_sync(ctx)))
      return fail(e);
  }
  *out = st;
  return GBS_OK;
}

gbs_status state_from_V(gbs_ctx* ctx, int M, const double* V, gbs_state** out) {
  if (M < 1 || !V || !out) return set_error(ctx, GBS_EINVAL, "gbs_state_from_V: bad arguments");
  const long long D = 2LL * M;
  gbs_state* st = nullptr;
  alloc_state(ctx, M, &st);
  DevBuf X, work;
  gbs_status e;
  auto fail = [&](gbs_status code) {
    dev_free(ctx, X);
    dev_free(ctx, work);
    gbs_state_free(st);
    return code;
  };
  // panels C and G, two inverses and a copy of a pivot block, then the pivots, and what the
  // host reads in one copy: their logarithms' sum, the status words and the row sums
  const size_t zc = 2 * (size_t)D * kSW + 3 * kSW * kSW, zd = 2 * (size_t)D + 2;
  if ((e = dev_alloc(ctx, st->V, D * D * 16)) || (e = dev_alloc(ctx, st->Sinv, D * D * 16)) ||
      (e = dev_alloc(ctx, X, D * D * 16)) || (e = dev_alloc(ctx, work, zc * 16 + zd * 8)))
    return fail(e);
  cudaStream_t s = ctx->stream;
  cplx<double>* x = (cplx<double>*)X.ptr;
  cplx<double>* C = (cplx<double>*)work.ptr;
  cplx<double>* G = C + D * kSW;
  cplx<double>* P[2] = {G + D * kSW, G + D * kSW + kSW * kSW};
  cplx<double>* Xk = P[1] + kSW * kSW;
  double* pv = (double*)(Xk + kSW * kSW);
  double* result = pv + D;
  int* status = (int*)(result + 1);  // [0] not positive definite, [1] not finite
  double* rowsum = result + 2;
  if ((e = check_cuda(ctx, cudaMemcpyAsync(st->V.ptr, V, D * D * 16, cudaMemcpyHostToDevice, s), "copy V")) ||
      (e = check_cuda(ctx, cudaMemsetAsync(status, 0, 2 * sizeof(int), s), "memset")))
    return fail(e);
  sigma_from_V_kernel<<<(unsigned)((D + 7) / 8), 256, 0, s>>>((const cplx<double>*)st->V.ptr, (int)D, x, rowsum, status + 1);
  sweep_first_kernel<<<1, 256, 0, s>>>(x, (int)D, P[0], pv, status);
  const int nb = (int)((D + kSW - 1) / kSW), ntiles = nb * (nb + 1) / 2;
  if (nb > 1) {
    for (int k = 0; k < nb; ++k) {
      sweep_panel_kernel<<<nb, 256, 0, s>>>(x, (int)D, k * kSW, P[k & 1], C, G, Xk);
      sweep_update_kernel<<<ntiles + (k + 1 < nb ? 1 : 0), 256, 0, s>>>(x, (int)D, k * kSW, ntiles, P[k & 1], C, G, Xk,
                                                                       P[(k + 1) & 1], pv, status);
    }
    count_launch(ctx, 2 * nb);
  }
  sweep_negate_kernel<<<(unsigned)((D * D + 255) / 256), 256, 0, s>>>(x, (int)D, (cplx<double>*)st->Sinv.ptr);
  sum_dd_kernel<true><<<1, 256, 0, s>>>(pv, (int)D, result);
  count_launch(ctx, 4);
  if ((e = check_cuda(ctx, cudaGetLastError(), "sigma inverse"))) return fail(e);
  std::vector<double> got(D + 2);
  if ((e = check_cuda(ctx, cudaMemcpyAsync(got.data(), result, (D + 2) * 8, cudaMemcpyDeviceToHost, s), "copy")) ||
      (e = stream_sync(ctx)))
    return fail(e);
  int hstatus[2];
  memcpy(hstatus, &got[1], sizeof hstatus);
  if (hstatus[1]) return fail(set_error(ctx, GBS_EINVAL, "gbs_state_from_V: non-finite V"));
  if (hstatus[0]) return fail(set_error(ctx, GBS_ENOTPD, "gbs_state_from_V: Sigma = V + I/2 is not positive definite"));
  st->logdet_sigma = got[0];
  // Gershgorin bound on the largest eigenvalue of Sigma = V + I/2
  for (long long i = 0; i < D; ++i) st->sigma_max = std::max(st->sigma_max, got[2 + i]);
  dev_free(ctx, X);
  dev_free(ctx, work);
  *out = st;
  return GBS_OK;
}

// Enqueue the packed click block (Sigma^-1)_S into dev_out.
gbs_status click_block(gbs_ctx* ctx, const gbs_state* st, const int* modes, int N, int real_basis, void* dev_out) {
  ModeList S;
  for (int i = 0; i < 32; ++i) S.m[i] = i < N ? modes[i] : 0;
  cudaStream_t s = ctx->stream;
  if (st->has_factors) {
    const int npairs = N * (N + 1) / 2;
    const int threads = 32 * npairs;
    sigma_inv_block_kernel<<<(threads + 255) / 256, 256, 0, s>>>(
        (const cplx<double>*)st->U.ptr, (const double*)st->alpha.ptr, (const double*)st->beta.ptr, st->M, S, N,
        real_basis, dev_out);
  } else {
    const int npairs = N * (N + 1) / 2;
    gather_inv_block_kernel<<<(npairs + 127) / 128, 128, 0, s>>>((const cplx<double>*)st->Sinv.ptr, st->M, S, N,
                                                                   real_basis, dev_out);
  }
  count_launch(ctx);
  return check_cuda(ctx, cudaGetLastError(), "click block");
}

}  // namespace gbs
