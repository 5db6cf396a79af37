// Device steps of the chain-rule sampler shared by its two drivers (a launch per step
// and operation, gbs_sampler.cu; whole steps in one CTA, gbs_chain.cu), so that both
// give the same bits: the root of a step's tree and the decision.
//
// Sigma' of a trajectory is kept in its lower triangle only (row >= column): the
// conditioning updates half the entries.  Modes are measured from the last one down, so
// a clicked mode's rows lie below the measured mode's, and those below the rest.
#pragma once
#include "gbs_internal.h"
#include "gbs_num.cuh"

namespace gbs {

// Entry (a, b) of Sigma', from the lower triangle.
__device__ __forceinline__ double sig_at(const double* sig, long long D, long long a, long long b) {
  return a >= b ? sig[a * D + b] : sig[b * D + a];
}

// The 2 x 2 pivot block of mode k and its inverse.
struct ModePivot {
  double det, q00, q10, q11;
};
__device__ __forceinline__ ModePivot mode_pivot(const double* sig, long long D, int k) {
  const long long r = 2LL * k;
  const double p00 = sig[r * D + r], p10 = sig[(r + 1) * D + r], p11 = sig[(r + 1) * D + r + 1];
  ModePivot m;
  m.det = fma(p00, p11, -(p10 * p10));
  const double inv = 1.0 / m.det;
  m.q00 = p11 * inv;
  m.q10 = -p10 * inv;
  m.q11 = p00 * inv;
  return m;
}

// Packed entry e of the root of a step's tree.  Full: Sigma'[S u {k}] with k last.
// Half: (Sigma'|k)[S], the Schur complement of mode k restricted to the clicked modes.
__device__ __forceinline__ double step_root(const double* sig, long long D, const int* clicks, int m, int k, bool half,
                                            const ModePivot& pv, int e) {
  int a = (int)((sqrtf(8.0f * e + 1.0f) - 1.0f) * 0.5f);
  while (a * (a + 1) / 2 > e) --a;
  while ((a + 1) * (a + 2) / 2 <= e) ++a;
  const int b = e - a * (a + 1) / 2;
  const int ma = (a >> 1) < m ? clicks[a >> 1] : k;
  const int mb = (b >> 1) < m ? clicks[b >> 1] : k;
  const long long ra = 2LL * ma + (a & 1), rb = 2LL * mb + (b & 1), rk = 2LL * k;
  double x = sig_at(sig, D, ra, rb);
  if (half) {
    const double ua0 = sig[ra * D + rk], ua1 = sig[ra * D + rk + 1];
    const double ub0 = sig[rb * D + rk], ub1 = sig[rb * D + rk + 1];
    const double l0 = fma(ua0, pv.q00, ua1 * pv.q10), l1 = fma(ua0, pv.q10, ua1 * pv.q11);
    x = fma(-l0, ub0, fma(-l1, ub1, x));
  }
  return x;
}

__device__ __forceinline__ double splitmix_u(unsigned long long seed, unsigned long long n) {
  unsigned long long z = seed + n * 0x9E3779B97F4A7C15ull;
  z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
  z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
  z ^= z >> 31;
  return (double)(z >> 11) * 0x1p-53;
}

// The decision of a step.  inc: the tree's Torontonian (half) or F_inc; exc: F_exc
// (full); dcarry: D of this step (half), replaced by the next step's when the mode stays
// dark.  p0 is formed in double-double: the quotient of the leading words and one
// correction from the exact residual (2^-100 relative before the last rounding) -- a
// triple-double quotient of two more steps gives the same double and took most of a
// 12 us kernel of dependent FP64 operations.
struct Decision {
  double p0;
  int click, near_tie;
};
__device__ __forceinline__ Decision decide_step(const double* inc, const double* exc, double* dcarry, bool half, int m,
                                                const ModePivot& pv, int forced, unsigned long long seed, int step,
                                                int sample, int attempt) {
  const double sgn = (m & 1) ? -1.0 : 1.0;  // (-1)^m
  td a, b, xnext;
  if (half) {
    xnext = td{inc[0] * sgn, inc[1] * sgn, inc[2] * sgn};  // (-1)^m Tor_k: D of the next step if k stays dark
    a = xnext * rsqrt(pv.det);
    b = td{dcarry[0], dcarry[1], dcarry[2]};
  } else {
    a = td{inc[0] * sgn, inc[1] * sgn, inc[2] * sgn};
    b = td{exc[0] * -sgn, exc[1] * -sgn, exc[2] * -sgn};
    xnext = a * sqrt(pv.det);  // Nn_k / det(P)^(-1/2)
  }
  const double ib = 1.0 / b.x0;
  const double q0 = a.x0 * ib;
  const double r = fma(-q0, b.x0, a.x0) + fma(-q0, b.x1, a.x1);
  Decision d;
  d.p0 = fma(r, ib, q0);
  d.near_tie = 0;
  if (forced >= 0) {
    d.click = forced;
  } else {
    const unsigned long long n =
        1ull + (unsigned long long)step + (1ull << 20) * ((unsigned long long)attempt + (1ull << 12) * (unsigned long long)sample);
    const double u = splitmix_u(seed, n);
    d.click = !(u < d.p0);
    d.near_tie = fabs(u - d.p0) < 1e-9;
  }
  if (!d.click) {
    dcarry[0] = xnext.x0;
    dcarry[1] = xnext.x1;
    dcarry[2] = xnext.x2;
  }
  return d;
}

}  // namespace gbs
