// Fixed-point multiword numbers on the integer pipe: the "FX" precisions.
//
// The subset tree needs ~160-bit arithmetic once the cancellation ratio passes
// ~1e20.  Built from FP64 error-free transformations (triple-double) each
// operation costs ~30 FP64 instructions, and this GPU issues only 2 FP64 FMAs
// per clock per SM, against ~60 32-bit integer multiply-adds and carry-chained
// adds.  fxn<L, F> holds a two's-complement integer X of L 32-bit limbs (limb 0
// least significant) read as X * 2^(-32 F).  Two widths serve each precision:
// the matrix entries and the scalars derived from them (pivots, determinants,
// inverse square roots) need only 31 integer bits, the running product s of
// pivot factors and the sums of terms need 63:
//   FXN   entries fxn4 = fxn<5, 4>, s and sums fxn4s = fxn<6, 4>  (128 fraction bits)
//   FX    entries fx   = fxn<6, 5>, s and sums fxs   = fxn<7, 5>  (160 fraction bits)
//   FXW   entries fxw  = fxn<7, 6>, s and sums fxws  = fxn<8, 6>  (192 fraction bits)
// Additions are exact (one carry-chained instruction per limb); a product
// keeps the columns at and above the fraction point of the exact 2L-limb
// product, which leaves an error of at most F units of the last place,
// biased low.
//
// Inside the tree every value stays in range when the caller has checked it:
// entries are bounded by the largest eigenvalue of the root, pivot
// determinants by its smallest, and s and the sums by (1 + 1/lambda_min)^n.
// A pivot determinant outside [2^-20, 2^12) is reported (kStatusRange) and
// the caller redoes the tree in triple-double.
//
// Everything here is device code; the host copies exist only so that the
// generic host/device helpers of the tree compile, and are never called.
#pragma once
#include <stdint.h>
#include <string.h>

#include "gbs_num.cuh"

namespace gbs {

template <int L, int F>
struct fxn {
  static_assert(F >= 2 && L > F, "at least two fraction limbs and one integer limb");
  uint32_t w[L];
};
typedef fxn<3, 2> fxd;   // FP64 trees of bounded states: entries (64 fraction bits)
typedef fxn<5, 2> fxds;  // their s and sums
typedef fxn<5, 4> fxn4;  // FXN entries
typedef fxn<6, 4> fxn4s; // FXN s and sums
typedef fxn<6, 5> fx;    // FX entries
typedef fxn<7, 5> fxs;   // FX s and sums
typedef fxn<7, 6> fxw;   // FXW entries
typedef fxn<8, 6> fxws;  // FXW s and sums

// ------------------------------------------------ carry-chained primitives --
// The carry flag lives between consecutive volatile asm statements of one
// chain; nothing else in these functions touches it.
#ifdef __CUDA_ARCH__
#define GBS_ASM1(op, r, a, b) asm volatile(op " %0, %1, %2;" : "=r"(r) : "r"(a), "r"(b))
#else
#define GBS_ASM1(op, r, a, b) (r = 0u)
#endif
GBS_HD uint32_t add_cc(uint32_t a, uint32_t b) { uint32_t r; GBS_ASM1("add.cc.u32", r, a, b); return r; }
GBS_HD uint32_t addc_cc(uint32_t a, uint32_t b) { uint32_t r; GBS_ASM1("addc.cc.u32", r, a, b); return r; }
GBS_HD uint32_t addc(uint32_t a, uint32_t b) { uint32_t r; GBS_ASM1("addc.u32", r, a, b); return r; }
GBS_HD uint32_t sub_cc(uint32_t a, uint32_t b) { uint32_t r; GBS_ASM1("sub.cc.u32", r, a, b); return r; }
GBS_HD uint32_t subc_cc(uint32_t a, uint32_t b) { uint32_t r; GBS_ASM1("subc.cc.u32", r, a, b); return r; }
GBS_HD uint32_t subc(uint32_t a, uint32_t b) { uint32_t r; GBS_ASM1("subc.u32", r, a, b); return r; }
#undef GBS_ASM1

// ---------------------------------------------------------------- basics --
template <int L, int F>
GBS_HD fxn<L, F> operator+(const fxn<L, F>& a, const fxn<L, F>& b) {
  fxn<L, F> r;
  r.w[0] = add_cc(a.w[0], b.w[0]);
#pragma unroll
  for (int k = 1; k < L - 1; ++k) r.w[k] = addc_cc(a.w[k], b.w[k]);
  r.w[L - 1] = addc(a.w[L - 1], b.w[L - 1]);
  return r;
}
template <int L, int F>
GBS_HD fxn<L, F> operator-(const fxn<L, F>& a, const fxn<L, F>& b) {
  fxn<L, F> r;
  r.w[0] = sub_cc(a.w[0], b.w[0]);
#pragma unroll
  for (int k = 1; k < L - 1; ++k) r.w[k] = subc_cc(a.w[k], b.w[k]);
  r.w[L - 1] = subc(a.w[L - 1], b.w[L - 1]);
  return r;
}
template <int L, int F>
GBS_HD fxn<L, F> operator-(const fxn<L, F>& a) {
  fxn<L, F> r;
  r.w[0] = sub_cc(0u, a.w[0]);
#pragma unroll
  for (int k = 1; k < L - 1; ++k) r.w[k] = subc_cc(0u, a.w[k]);
  r.w[L - 1] = subc(0u, a.w[L - 1]);
  return r;
}
// ---------------------------------------------------------------- product --
// out[0 .. CHI - CLO] receives columns CLO .. CHI (32-bit words of weight
// 2^(32 c)) of the sum of the partial products a_i b_j with i + j in
// [CLO, CHI] of two unsigned multiword integers, modulo 2^(32 (CHI + 1)).
//
// What bounds a product is the multiply pipe: a 32 x 32 + 64 bit multiply-add
// holds it for about 4 cycles per warp.  A partial product is a pair of words;
// pairs that start at columns of equal parity never overlap, so each row of
// partial products is two carry chains (even and odd columns) of mad.lo.cc /
// madc.hi.cc pairs, each pair being one wide multiply-add with carry in and out
// and nothing else; the two accumulators are added once at the end.  A chain's
// last carry goes to the next pair of its parity, which no earlier row has
// reached (rows go up, and so do their ends), so it never carries further.
// Measured on the GB300 (chains of dependent 26-partial-product products, 16
// warps per SM): 42.5 instructions per product, multiply pipe 90 % busy, 322 G/s,
// against 97 instructions, 80 % and 219 G/s for 64-bit multiply-adds with a
// separate running carry (78 adds and moves beside the 26 multiplies).
#ifdef __CUDA_ARCH__
#define GBS_ASM3(op, r, a, b, c) asm volatile(op " %0, %1, %2, %3;" : "=r"(r) : "r"(a), "r"(b), "r"(c))
#else
#define GBS_ASM3(op, r, a, b, c) (r = 0u)
#endif
GBS_HD uint32_t mad_lo_cc(uint32_t a, uint32_t b, uint32_t c) { uint32_t r; GBS_ASM3("mad.lo.cc.u32", r, a, b, c); return r; }
GBS_HD uint32_t madc_lo_cc(uint32_t a, uint32_t b, uint32_t c) { uint32_t r; GBS_ASM3("madc.lo.cc.u32", r, a, b, c); return r; }
GBS_HD uint32_t madc_hi_cc(uint32_t a, uint32_t b, uint32_t c) { uint32_t r; GBS_ASM3("madc.hi.cc.u32", r, a, b, c); return r; }
#undef GBS_ASM3

// UPPER: only the partial products with j > i (the half of a square).
template <int NA, int NB, int CLO, int CHI, bool UPPER = false>
GBS_HD void prod_cols(const uint32_t* a, const uint32_t* b, uint32_t* out) {
  uint32_t acc[2][CHI + 4];
#pragma unroll
  for (int k = 0; k < CHI + 4; ++k) acc[0][k] = acc[1][k] = 0u;
#pragma unroll
  for (int i = 0; i < NA; ++i) {
#pragma unroll
    for (int p = 0; p < 2; ++p) {
      int end = -1;
#pragma unroll
      for (int j = 0; j < NB; ++j) {
        const int c = i + j;
        if (c < CLO || c > CHI || (c & 1) != p || (UPPER && j <= i)) continue;
        acc[p][c] = end < 0 ? mad_lo_cc(a[i], b[j], acc[p][c]) : madc_lo_cc(a[i], b[j], acc[p][c]);
        if (c < CHI) acc[p][c + 1] = madc_hi_cc(a[i], b[j], acc[p][c + 1]);
        end = c;
      }
      if (end >= 0 && i > 0 && end + 2 <= CHI) acc[p][end + 2] = addc(acc[p][end + 2], 0u);
    }
  }
  // column CLO holds one accumulator only
  constexpr int P = CLO & 1;
  out[0] = acc[P][CLO];
  if constexpr (CHI > CLO) {
    out[1] = add_cc(acc[0][CLO + 1], acc[1][CLO + 1]);
#pragma unroll
    for (int c = CLO + 2; c < CHI; ++c) out[c - CLO] = addc_cc(acc[0][c], acc[1][c]);
    if constexpr (CHI > CLO + 1) out[CHI - CLO] = addc(acc[0][CHI], acc[1][CHI]);
  }
}

// a * b of non-negative values (a with LA limbs, the result too): the columns
// from the fraction point up, formed with one guard column below it whose sum is
// dropped: at most F units of the last place, always toward -inf.  Every product
// of the tree is of this kind: a signed factor is shifted by a power of two first
// (one add in its integer limb), and the shift's effect is separable and folded
// into constants (fx_pivot below).  A two's-complement correction instead costs
// 20-25 adds and masks a product (259 against 322 G products/s).
template <int LA, int LB, int F>
GBS_HD fxn<LA, F> umul(const fxn<LA, F>& a, const fxn<LB, F>& b) {
  uint32_t t[LA + 1];
  prod_cols<LA, LB, F - 1, F + LA - 1>(a.w, b.w, t);
  fxn<LA, F> r;
#pragma unroll
  for (int k = 0; k < LA; ++k) r.w[k] = t[k + 1];
  return r;
}

// a * a of a non-negative value: the products of two different limbs once, doubled,
// then the limbs' squares in one carry chain (15 partial products for F = 5, against
// 26).  The error is that of umul.
template <int L, int F>
GBS_HD fxn<L, F> usqr(const fxn<L, F>& a) {
  constexpr int CLO = F - 1, CHI = F + L - 1;
  uint32_t t[CHI - CLO + 1];
  prod_cols<L, L, CLO, CHI, true>(a.w, a.w, t);
#pragma unroll
  for (int k = CHI - CLO; k > 0; --k) t[k] = (t[k] << 1) | (t[k - 1] >> 31);
  t[0] <<= 1;
  bool first = true;
#pragma unroll
  for (int i = (CLO + 1) / 2; i < L && 2 * i <= CHI; ++i) {
    uint32_t& lo = t[2 * i - CLO];
    lo = first ? mad_lo_cc(a.w[i], a.w[i], lo) : madc_lo_cc(a.w[i], a.w[i], lo);
    if (2 * i < CHI) t[2 * i + 1 - CLO] = madc_hi_cc(a.w[i], a.w[i], t[2 * i + 1 - CLO]);
    first = false;
  }
  fxn<L, F> r;
#pragma unroll
  for (int k = 0; k < L; ++k) r.w[k] = t[k + 1];
  return r;
}

// ----------------------------------------------------------- conversions --
// Exact while |x| fits the integer limbs, down to 2^-(32 F) (bits below are
// dropped, toward zero).
template <int L, int F>
GBS_HD fxn<L, F> fx_from_double(double x) {
  fxn<L, F> r;
#ifdef __CUDA_ARCH__
  const unsigned long long bits = (unsigned long long)__double_as_longlong(x);
#else
  unsigned long long bits;
  memcpy(&bits, &x, 8);
#endif
  const int e = (int)((bits >> 52) & 0x7ff);
  const unsigned long long m = (bits & 0xfffffffffffffull) | (e ? (1ull << 52) : 0ull);
  const int sh = (e ? e : 1) - 1075 + 32 * F;  // bit position of m's last bit in X
#pragma unroll
  for (int k = 0; k < L; ++k) {
    const int s = 32 * k - sh;
    const unsigned long long v = s >= 0 ? (s < 64 ? (m >> s) : 0ull) : (s > -64 ? (m << (-s)) : 0ull);
    r.w[k] = (uint32_t)v;
  }
  return (bits >> 63) ? -r : r;
}
template <int L, int F>
GBS_HD fxn<L, F> fx_of_(double x, fxn<L, F>*) {
  return fx_from_double<L, F>(x);
}
// x as the fixed-point type E.
template <class E>
GBS_HD E fx_of(double x) {
  return fx_of_(x, (E*)nullptr);
}

// Nearest-ish double (a few units of the last place).
template <int L, int F>
GBS_HD double to_double(const fxn<L, F>& a) {
  double v = (double)(int32_t)a.w[L - 1];
#pragma unroll
  for (int k = L - 2; k >= 0; --k) v = fma(v, 4294967296.0, (double)a.w[k]);
  return v * (F == 2 ? 0x1p-64 : F == 4 ? 0x1p-128 : F == 5 ? 0x1p-160 : 0x1p-192);
}
static_assert(sizeof(fxn4) == 20 && sizeof(fxn4s) == 24 && sizeof(fx) == 24 && sizeof(fxs) == 28 &&
                  sizeof(fxw) == 28 && sizeof(fxws) == 32,
              "fx widths");

// The s type (running product of pivot factors, term sums) of an entry type.
template <class E> struct fx_sum;
template <> struct fx_sum<fxd> { typedef fxds type; };
template <> struct fx_sum<fxn4> { typedef fxn4s type; };
template <> struct fx_sum<fx> { typedef fxs type; };
template <> struct fx_sum<fxw> { typedef fxws type; };

// A pivot determinant the fixed-point tree can use: in [2^-20, 2^12), where
// its inverse square root keeps ~150 bits (the resolution is absolute, so the
// relative error of 1/sqrt(x) grows like 2^-(32 F) x).
template <int L, int F>
GBS_HD bool fx_det_in_range(const fxn<L, F>& d) {
  bool high_zero = true;
#pragma unroll
  for (int k = F + 1; k < L; ++k) high_zero &= d.w[k] == 0u;
  return high_zero && d.w[F] < (1u << 12) && (d.w[F] != 0u || d.w[F - 1] >= (1u << 12));
}

// 1/sqrt(x) for x in [2^-20, 2^12), on the integer pipe apart from an FP32 seed.
// x is normalised to x = m 2^(2h), m in [1, 4), as the integer M = m 2^(32 F + 30)
// of F + 1 limbs (so its top limb has two integer bits), and y = m^(-1/2) in
// (1/2, 1] is refined by third-order steps y <- y (1 + e/2 + 3 e^2/8), e = 1 - m y^2:
//   seed   the single-precision inverse square root of the float of M's top limb,
//          Y0 = y0 2^31, |e| < 2^-20; if y0 rounded to 12 significant bits squares
//          exactly to 1/m in single precision it is taken instead, so that exact
//          cases (x = 1, 1/4, 4, ...) stay exact;
//   1.     e 2^64 from the exact 128-bit difference 2^124 - (top 64 bits of M) Y0^2;
//          Y1 = y1 2^63 (64 bits), |e| < 2^-59;
//   2.     (F > 2) e from the product of M and the exact 128-bit Y1^2, of which only
//          the columns from just below the wanted resolution up to the one |e| can
//          reach are formed (the leading ones cancel against the 1); e^2 from the
//          top 64 bits of e; the result's relative error is below 2^-165 (F >= 5),
//          2^-150 (F = 4).
// With F = 2 the value after step 1 is returned (relative error below 2^-61).
// The normalisation makes every factor short: 39 partial products for F = 5,
// against 89 for the same steps on the unnormalised limbs.
template <int L, int F>
__device__ __forceinline__ fxn<L, F> rsqrt_(const fxn<L, F>& x) {
  static_assert(L == F + 1, "one integer limb");
  const unsigned long long top = ((unsigned long long)x.w[F] << 32) | x.w[F - 1];
  const int sh = __clzll((long long)top) & ~1;  // 20 .. 50 (garbage in, garbage out beyond)
  const bool mv = sh >= 32;
  uint32_t M[F + 1];  // x's limbs << sh
#pragma unroll
  for (int k = F; k >= 0; --k) {
    const uint32_t hi = mv ? (k >= 1 ? x.w[k >= 1 ? k - 1 : 0] : 0u) : x.w[k];
    const uint32_t lo = mv ? (k >= 2 ? x.w[k >= 2 ? k - 2 : 0] : 0u) : (k >= 1 ? x.w[k >= 1 ? k - 1 : 0] : 0u);
    M[k] = __funnelshift_l(lo, hi, sh);
  }
  const int h = (30 - sh) / 2;  // -10 .. 5 (sh is even)
  const float mf = __uint2float_rn(M[F]) * 0x1p-30f;
  float yf = rsqrtf(mf);
  const float ys = __uint_as_float((__float_as_uint(yf) + 0x800u) & ~0xfffu);
  if (fmaf(mf * ys, ys, -1.0f) == 0.0f) yf = ys;
  const uint32_t Y0 = __float2uint_rz(yf * 0x1p31f);
  // step 1
  const unsigned long long q0 = (unsigned long long)Y0 * Y0;
  const unsigned long long mt = ((unsigned long long)M[F] << 32) | M[F - 1];
  const unsigned long long plo = mt * q0, phi = __umul64hi(mt, q0);
  const unsigned long long dhi = (1ull << 60) - phi - (plo != 0ull);
  const long long e64 = (long long)((dhi << 4) | ((0ull - plo) >> 60));  // e 2^64
  const int es = (int)(e64 >> 14);                                       // e 2^50
  const unsigned long long sq = (unsigned long long)((long long)es * es) >> 36;
  const long long f = (e64 >> 1) + (long long)((sq * 3ull) >> 3);        // (e/2 + 3 e^2/8) 2^64
  const int fh = (int)(f >> 32);
  const unsigned long long Y1 = ((unsigned long long)Y0 << 32) + (unsigned long long)((long long)fh * (long long)Y0) +
                                (((unsigned long long)(uint32_t)f * Y0) >> 32);
  fxn<L, F> r;
  const uint32_t yh = (uint32_t)(Y1 >> 32), yl = (uint32_t)Y1;
  if constexpr (F == 2) {
    // y 2^(64 + 26), then down by 26 + h (16 .. 31)
    const uint32_t a0 = yl << 27, a1 = __funnelshift_l(yl, yh, 27), a2 = yh >> 5;
    r.w[0] = __funnelshift_r(a0, a1, 26 + h);
    r.w[1] = __funnelshift_r(a1, a2, 26 + h);
    r.w[2] = a2 >> ((26 + h) & 31);
    return r;
  } else {
    // step 2
    const unsigned long long ll = (unsigned long long)yl * yl, lh = (unsigned long long)yl * yh,
                             hh = (unsigned long long)yh * yh;
    const unsigned long long s0 = ll + (lh << 33);
    const unsigned long long s1 = hh + (lh >> 31) + (s0 < ll ? 1ull : 0ull);
    const uint32_t q[4] = {(uint32_t)s0, (uint32_t)(s0 >> 32), (uint32_t)s1, (uint32_t)(s1 >> 32)};
    // 1 = 2^(32 F + 156) in the product; e needs the columns CLO + 1 .. CHI
    constexpr int CHI = (32 * F + 156 - 59) / 32;
    constexpr int CLO = F >= 6 ? 4 : 3;
    constexpr int NE = CHI - CLO;  // limbs of e 2^U2
    uint32_t t[NE + 1];
    prod_cols<F + 1, 4, CLO, CHI>(M, q, t);
    uint32_t e[NE];
    e[0] = sub_cc(0u, t[1]);
#pragma unroll
    for (int k = 1; k < NE - 1; ++k) e[k] = subc_cc(0u, t[k + 1]);
    e[NE - 1] = subc(0u, t[NE]);
    // c = e/2 + 3 e^2/8 in units of 2^-U, U = 32 F + 155 - 32 (CLO + 1); |c| < 2^-60
    constexpr int NC = NE - 1;  // limbs of c, two's complement
    uint32_t c[NC];
#pragma unroll
    for (int k = 0; k < NC; ++k) c[k] = __funnelshift_r(e[k], e[k + 1], 2);
    const uint32_t neg = (uint32_t)((int32_t)c[NC - 1] >> 31);
    // |e/2| 2^(U - 32 (NC - 2)) in two limbs (the truncated rest is below 2^-123)
    const uint32_t ah = c[NC - 1] ^ neg, al = c[NC - 2] ^ neg;
    const unsigned long long sll = (unsigned long long)al * al, slh = (unsigned long long)al * ah,
                             shh = (unsigned long long)ah * ah;
    const unsigned long long sm = (sll >> 32) + (slh << 1);  // (2 al ah) + carry: below 2^64 as ah < 2^31
    const unsigned long long sq2 = shh + (sm >> 32);         // (e/2)^2 2^(2U - 64 (NC - 2) - 64)
    // (e/2)^2 in units of 2^-U: up by U - (2U - 64 (NC - 2) - 64) = 64 (NC - 1) - U
    constexpr int U = 32 * F + 155 - 32 * (CLO + 1);
    constexpr int DN = U - 64 * (NC - 1);  // -5 (F = 5, 6) or 27 (F = 4)
    static_assert(DN == -5 || DN == 27, "alignment of the squared residual");
    unsigned long long q2;
    uint32_t q2h;
    if constexpr (DN == -5) {
      const unsigned long long w = (sq2 << 5) | ((sm & 0xffffffffull) >> 27);
      const uint32_t wh = (uint32_t)(sq2 >> 59);
      q2 = w + ((w >> 1) | ((unsigned long long)wh << 63));  // 3/2 (e/2)^2
      q2h = wh + (wh >> 1) + (q2 < w ? 1u : 0u);
    } else {
      const unsigned long long w = sq2 >> 27;
      q2 = w + (w >> 1);
      q2h = 0u;
    }
    c[0] = add_cc(c[0], (uint32_t)q2);
    c[1] = addc_cc(c[1], (uint32_t)(q2 >> 32));
    if constexpr (NC == 3) {
      c[2] = addc(c[2], q2h);
    } else {
      c[2] = addc_cc(c[2], q2h);
#pragma unroll
      for (int k = 3; k < NC - 1; ++k) c[k] = addc_cc(c[k], 0u);
      c[NC - 1] = addc(c[NC - 1], 0u);
    }
    // y 2^(U - 1) = Y1 2^(U - 64) + c Y1 2^-64 (NC + 2 limb product, limbs 2 up)
    const uint32_t sg = (uint32_t)((int32_t)c[NC - 1] >> 31);
    const uint32_t yy[2] = {yl, yh};
    uint32_t d[NC + 1];
    prod_cols<NC, 2, 1, NC + 1>(c, yy, d);  // d[k]: limb k + 1; d[0] is the guard
    uint32_t o[NC + 1];                      // limbs 2 .. NC + 1, then the sign
#pragma unroll
    for (int k = 0; k < NC; ++k) o[k] = d[k + 1];
    o[NC - 2] = sub_cc(o[NC - 2], yl & sg);
    o[NC - 1] = subc_cc(o[NC - 1], yh & sg);
    // Y1 2^(U - 64) covers the limbs Z .. Z + 2
    constexpr int ZB = U - 64, Z = ZB / 32, ZS = ZB % 32;
    constexpr int NO = NC + 2;
    uint32_t z[NO];
#pragma unroll
    for (int k = 0; k < NO; ++k) z[k] = 0u;
    z[Z] = yl << ZS;
    z[Z + 1] = __funnelshift_l(yl, yh, ZS);
    z[Z + 2] = ZS ? yh >> (32 - ZS) : 0u;
    const uint32_t sx = (uint32_t)((int32_t)o[NC - 1] >> 31);
    uint32_t v[NO];
    v[0] = add_cc(z[0], o[0]);
#pragma unroll
    for (int k = 1; k < NO - 1; ++k) v[k] = addc_cc(z[k], k < NC ? o[k] : sx);
    v[NO - 1] = addc(z[NO - 1], sx);
    // v = y 2^(U - 1); the result is y 2^-h in units of 2^-32F: down by U - 1 - 32 F + h
    constexpr int SD = U - 1 - 32 * F;  // 26 (F <= 5) or -6 (F = 6: one limb of zeros below)
    static_assert(SD == 26 || SD == -6, "alignment of the result");
    constexpr int PADL = SD < 0 ? 1 : 0;
#pragma unroll
    for (int k = 0; k < L; ++k) {
      const int a = k - PADL, b = a + 1;
      const uint32_t lo = a >= 0 && a < NO ? v[a >= 0 && a < NO ? a : 0] : 0u;
      const uint32_t hi = b >= 0 && b < NO ? v[b >= 0 && b < NO ? b : 0] : 0u;
      r.w[k] = __funnelshift_r(lo, hi, 26 + h);
    }
    return r;
  }
}

// Three doubles whose sum is the value to ~2^-159 relative (each the nearest
// double of what the previous ones left over; the differences are exact).
template <int L, int F>
GBS_HD void fx_store3(const fxn<L, F>& a, double* o) {
  const double x0 = to_double(a);
  const fxn<L, F> r1 = a - fx_from_double<L, F>(x0);
  const double x1 = to_double(r1);
  const fxn<L, F> r2 = r1 - fx_from_double<L, F>(x1);
  o[0] = x0;
  o[1] = x1;
  o[2] = to_double(r2);
}
template <int L, int F>
__device__ __forceinline__ fxn<L, F> shfl_down(const fxn<L, F>& v, int off) {
  fxn<L, F> r;
#pragma unroll
  for (int k = 0; k < L; ++k) r.w[k] = __shfl_down_sync(0xffffffffu, v.w[k], off);
  return r;
}

template <int L, int F>
__device__ __forceinline__ fxn<L, F> shfl_xor(const fxn<L, F>& v, int mask) {
  fxn<L, F> r;
#pragma unroll
  for (int k = 0; k < L; ++k) r.w[k] = __shfl_xor_sync(0xffffffffu, v.w[k], mask);
  return r;
}

}  // namespace gbs
