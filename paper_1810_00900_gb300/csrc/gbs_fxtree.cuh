// Subset-determinant trees in fixed point (gbs_fx.cuh): kernels.
//
// The decision tree of gbs_tree.cuh for the integer entry types, organised so
// that only *included* children are ever computed or stored: excluding a mode
// drops two rows, so an excluded child is a view of its parent's matrix.
//
// Nodes.  With the first D = n - Q modes of a tree decided, node v in [0, 2^D)
// has mode j included iff bit j of v is set.  Its matrix is that of its last
// included mode: v = 0 is the root (all n modes), and v with top bit k is matrix
// v - 2^k of level k, the Schur complement of the q = n - 1 - k modes after mode
// k given the included ones; a node at depth d > k is the trailing 2 (n - d) rows
// of it.  Level k has 2^k matrices, and its parents are exactly the nodes
// 0 .. 2^k - 1: matrix c of level k includes mode k at node c.  Against storing
// both children of every node this halves the writes and takes a quarter off the
// traffic.
//
//   top kernel    one CTA per node v < 2^dtop: eliminates the modes of v from the
//                 root in shared memory and writes that matrix; replaces the
//                 first levels, where nodes are few.
//   level kernels one launch per child size q: a warp per 32 consecutive children of a
//                 tree (lane = child), or, where children are few, a CTA per 1 .. 32.
//   leaf kernel   a warp takes tiles of 32 nodes of one tree, one thread per node
//                 for all 2^Q subsets of its last Q modes; a sum per CTA.
//   final kernel  one CTA per tree adds the CTAs' sums and finishes the result.
//   small kernel  a tree of few modes in one launch, in the shared memory of one or a
//                 few CTAs.
// Measured against the engine it replaced (both children stored, subtrees of 9
// modes expanded in shared memory, signed products, 2 products per entry), with the
// default launch shapes: N = 24 (M = 200, AUTO) 8.86 -> 2.4 ms, 256 requests of N =
// 8 .. 20 23.0 -> 6.7 ms.
// All sums are exact integers, and every pivot, row and entry is formed by the
// same functions below wherever it is formed: results do not depend on the launch
// shape or on the rest of the batch, bit for bit.
//
// Including a mode with pivot block P = [[p00, p10], [p10, p11]] and its columns
// U = (u0, u1): C' = C - L U^T, L = U P^-1.  Products are the cost, so they are
// saved where exact additions can take their place:
//   rows     the second pivot coordinate is flipped where p10 > 0, so that with
//            al = p11/det, be = p00/det, m = |p10|/det >= 0
//              L0 = (al + m) u0 - m (u0 - u1),  L1 = (be + m) u1 + m (u0 - u1):
//            three products per row in place of four;
//   entries  Winograd's inner product (S. Winograd, IEEE Trans. Comp. C-17, 1968):
//              L0_a u0_b + L1_a u1_b = (L0_a + u1_b)(u0_b + L1_a) - L0_a L1_a - u0_b u1_b:
//            one product per entry and two per row in place of two per entry.
// An update of R rows takes R (R + 1) / 2 + 5 R products in place of R (R + 1) +
// 4 R (R = 4, 6, 8: 30, 51, 76 for 36, 66, 104).  Neither form loses accuracy
// here: sums are exact and a product's error is absolute, whatever its factors.
// Signed factors are shifted by K = 2^29, so that all products are of
// non-negative values; the shifts are separable and live in c0, c1, A and B:
//   U = u0 + K, V = u1 + K, P = L0 + K, Q = L1 + K
//   P = (al + m) U - m (U - V + 2K) + c0,  c0 = K + 2K m - K (al + m)
//   Q = (be + m) V + m (U - V + 2K) + c1,  c1 = K - 2K m - K (be + m)
//   A = (P + K)(Q + K) - 2 K^2,  B = (U + K)(V + K) - 2 K^2
//   C' = C - (P_a + V_b)(U_b + Q_a) + A_a + B_b
// All of it holds modulo 2^32, the range of the integer limb, so only the factors need a
// bound: |u| and |L| below K.  K costs no accuracy: it lies in the integer limb, whose
// partial products are all kept, so the bits do not depend on it.  The roots are checked
// (fx_root_entry_ok, fx_root_mode_ok): entries below 2^29, and by positive definiteness all
// entries of the tree; and the product of a mode's diagonal entries below 2^31, so that no
// determinant wraps past the check of its range.  A row of L is bounded by |L_a|^2 <= C_aa
// lambda_max(P^-1): below 2^20 over (Sigma^-1)_S, whose eigenvalues are at least 1 / sigma_max
// >= 2^-10 whether V is physical or not, and below 2^17 over a conditioned Sigma', with
// entries up to 64 and det P >= 2^-20.  (K = 2^9, enough where Sigma >= I/2, lost states
// given by a V whose Sigma has eigenvalues down to 1/2000.)
#pragma once
#include "gbs_fx.cuh"
#include "gbs_internal.h"
#include "gbs_batch.cuh"

namespace gbs {

constexpr int kFxShiftBits = 29;
constexpr uint32_t kFxShift = 1u << kFxShiftBits;  // K

// Programmatic dependent launch: the launch after this one may set up its CTAs from
// here on; wait for the launch before this one to be complete.  Every thread of a kernel of
// the chain calls it before it touches memory that an earlier launch of the chain writes.
// Only the plan (segs, trees, lvl_off), uploaded before the chain's first launch, may be read
// ahead of it, and only the plan's pointers are const __restrict__: nodes, s, partial sums
// and status change while such a kernel is already running, so a load from them must not be
// taken for one of memory that is read-only throughout, which a compiler may move above the
// wait or through the non-coherent path.
__device__ __forceinline__ void fx_after() {
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  asm volatile("griddepcontrol.wait;" ::: "memory");
}

// Whether a root fits the engine (see above): |x| < 2^29 for every entry (NaN and infinities
// are not), and p00 p11 < 2^31 for every mode, from the integer limbs of its diagonal.
__device__ __forceinline__ bool fx_root_entry_ok(double x) {
  return (__double2hiint(x) & 0x7fffffff) < ((1023 + 29) << 20);
}
template <int L, int F>
__device__ __forceinline__ bool fx_root_mode_ok(const fxn<L, F>& p00, const fxn<L, F>& p11) {
  return ((unsigned long long)p00.w[L - 1] + 1ull) * ((unsigned long long)p11.w[L - 1] + 1ull) <= (1ull << 31);
}

// Scalars of a pivot.
template <class E>
struct FxPivot {
  E g, a, b, m, c0, c1;  // det^(-1/2), al + m, be + m, m and the row constants
  uint32_t flip;         // all ones: the second coordinate changes sign
};
// A row of the update: P, Q, A (as row a) and U, V, B (as column b).
template <class E>
struct FxRow {
  E P, Q, A, U, V, B;
};

// x + v 2^(32 F): v in the integer limb.
template <int L, int F>
GBS_HD fxn<L, F> fx_add_int(fxn<L, F> x, uint32_t v) {
  x.w[L - 1] += v;
  return x;
}
// x << s (0 < s < 32)
template <int L, int F>
__device__ __forceinline__ fxn<L, F> fx_shl(const fxn<L, F>& x, int s) {
  fxn<L, F> r;
#pragma unroll
  for (int k = L - 1; k > 0; --k) r.w[k] = __funnelshift_l(x.w[k - 1], x.w[k], s);
  r.w[0] = x.w[0] << s;
  return r;
}
// x, or -x where mask is all ones
template <int L, int F>
GBS_HD fxn<L, F> fx_flip(const fxn<L, F>& x, uint32_t mask) {
  fxn<L, F> t, r;
#pragma unroll
  for (int k = 0; k < L; ++k) t.w[k] = x.w[k] ^ mask;
  r.w[0] = sub_cc(t.w[0], mask);
#pragma unroll
  for (int k = 1; k < L - 1; ++k) r.w[k] = subc_cc(t.w[k], mask);
  r.w[L - 1] = subc(t.w[L - 1], mask);
  return r;
}

// |x|; mask (all ones where x < 0)
template <int L, int F>
GBS_HD fxn<L, F> fx_abs(const fxn<L, F>& x, uint32_t& mask) {
  mask = (uint32_t)((int32_t)x.w[L - 1] >> 31);
  return fx_flip(x, mask);
}

// det(P); the determinant alone is what a one-mode node needs.
template <class E>
__device__ __forceinline__ E fx_det(const E& p00, const E& p10, const E& p11) {
  uint32_t neg;
  const E n10 = fx_abs(p10, neg);
  return umul(p00, p11) - usqr(n10);
}

// Returns whether the determinant is in range.
template <class E>
__device__ __forceinline__ bool fx_pivot(const E& p00, const E& p10, const E& p11, FxPivot<E>& pv) {
  uint32_t neg;
  const E n10 = fx_abs(p10, neg);
  bool zero = true;
#pragma unroll
  for (int k = 0; k < (int)(sizeof(E) / 4); ++k) zero &= p10.w[k] == 0u;
  pv.flip = (neg == 0u && !zero) ? 0xffffffffu : 0u;  // p10 > 0
  const E det = umul(p00, p11) - usqr(n10);
  pv.g = rsqrt_(det);
  const E inv = usqr(pv.g);
  pv.m = umul(n10, inv);
  pv.a = umul(p11, inv) + pv.m;
  pv.b = umul(p00, inv) + pv.m;
  const E km = fx_shl(pv.m, kFxShiftBits + 1);  // 2 K m
  pv.c0 = fx_add_int(km - fx_shl(pv.a, kFxShiftBits), kFxShift);
  pv.c1 = fx_add_int(-(km + fx_shl(pv.b, kFxShiftBits)), kFxShift);
  return fx_det_in_range(det);
}

template <class E>
__device__ __forceinline__ void fx_row(const FxPivot<E>& pv, const E& u0, const E& u1, FxRow<E>& r) {
  r.U = fx_add_int(u0, kFxShift);
  r.V = fx_add_int(fx_flip(u1, pv.flip), kFxShift);
  const E mt = umul(pv.m, fx_add_int(r.U - r.V, 2 * kFxShift));
  r.P = umul(pv.a, r.U) - mt + pv.c0;
  r.Q = umul(pv.b, r.V) + mt + pv.c1;
  r.A = fx_add_int(umul(fx_add_int(r.P, kFxShift), fx_add_int(r.Q, kFxShift)), 0u - 2u * kFxShift * kFxShift);
  r.B = fx_add_int(umul(fx_add_int(r.U, kFxShift), fx_add_int(r.V, kFxShift)), 0u - 2u * kFxShift * kFxShift);
}

// Entry (a, b) of the child.
template <class E>
__device__ __forceinline__ E fx_entry(const E& c, const E& Pa, const E& Qa, const E& Aa, const E& Ub, const E& Vb,
                                      const E& Bb) {
  return (c + Aa + Bb) - umul(Pa + Vb, Ub + Qa);
}

// ------------------------------------------------------------- node buffers --
// Matrices of level k are packed lower triangles.  From level 5 on they lie in
// tiles of 32: limb l of entry e of matrix c is word ((c / 32) ne + e) 32 L + 32 l +
// c % 32, so a warp's access is one 128-byte line and the limbs of an entry are at
// constant distances (immediate offsets).  The root and levels 0 .. 4, less than a
// tile each, are stored one matrix after another (stride 1 between limbs).
template <class E, int ST>
__device__ __forceinline__ E fx_ld(const uint32_t* p, int e) {
  constexpr int L = sizeof(E) / 4;
  const uint32_t* q = p + (long long)e * (L * ST);
  E r;
#pragma unroll
  for (int k = 0; k < L; ++k) r.w[k] = q[k * ST];
  return r;
}
template <class E, int ST>
__device__ __forceinline__ void fx_st(uint32_t* p, int e, const E& v) {
  constexpr int L = sizeof(E) / 4;
  uint32_t* q = p + (long long)e * (L * ST);
#pragma unroll
  for (int k = 0; k < L; ++k) q[k * ST] = v.w[k];
}

// One tree of a batch.  Level k of it starts at word lvl_off[tab + k + 1] of the
// node buffer (k = -1: the root).
//
// A tree whose levels would not fit the workspace is taken in chunks: the nodes of
// depth d0 stay, and the levels from d0 on hold the descendants of 2^cb consecutive
// ones at a time.  Inside chunk h, index v' >= 2^cb stands for the node with low
// bits (v' mod 2^cb) + h 2^cb and its bits from d0 on those of v' from cb on; v' <
// 2^cb for node v' + h 2^cb of depth d0.  Unchunked, cb = d0 = 0 and v' = v.
// s of it is element s_base + v (v < 2^d0), s_base + 2^d0 - 2^cb + v'.
struct FxTree {
  long long root_off, s_base;
  double scale;  // det(Sigma)^(-1/2)
  int n, D, tree, tab, d0, cb;
};
struct FxSeg {
  long long first;  // first CTA (top) / tile (level) / warp unit (leaf) of this tree
  int idx, tiles_per_unit;
};
template <class Sum>
struct FxPart {
  Sum inc, exc, abs;
};

// The last segment that begins at or before key, by whole warps: 32 at a time, so that a
// launch over up to 32 trees waits for one load where a bisection waits for five.  (With
// the plan read before fx_after: 300 trees of 12 modes, 160 bits, 853 -> 828 us, 24 of 17
// 688 -> 672.)
__device__ __forceinline__ int fx_find(const FxSeg* segs, int n, long long key) {
  const int lane = threadIdx.x & 31;
  int lo = 0, step = 1;
  while (step * 32 < n) step *= 32;
  for (; step > 0; step /= 32) {
    const int i = lo + lane * step;
    const unsigned m = __ballot_sync(0xffffffffu, i < n && segs[i].first <= key);
    lo += (31 - __clz((int)(m | 1u))) * step;
  }
  return lo;
}

// Where the matrix of index v is, and how many modes (p) it holds.  ST = 32 for
// nodes in tiles, 1 for nodes 0 .. 31 of a tree.
template <int ST, int L>
__device__ __forceinline__ const uint32_t* fx_node(const uint32_t* nodes, const long long* lvl_off, const FxTree& t,
                                                   unsigned v, unsigned chunk, int& p) {
  int up = 0;  // levels of the tree above bit 0 of v's level
  if (v < (1u << t.cb)) {
    v += chunk << t.cb;
    if (v == 0u) {
      p = t.n;
      return nodes + lvl_off[t.tab];
    }
  } else {
    up = t.d0 - t.cb;
  }
  const int k = 31 - __clz((int)v);
  const unsigned c = v - (1u << k);
  p = t.n - 1 - k - up;
  const int ne = sym(2 * p);
  const uint32_t* base = nodes + lvl_off[t.tab + k + up + 1];
  if constexpr (ST == 1) return base + (long long)c * ne * L;
  return base + (long long)(c >> 5) * ne * (L * 32) + (c & 31u);
}
__device__ __forceinline__ long long fx_sidx(const FxTree& t, unsigned v, unsigned chunk) {
  return v < (1u << t.cb) ? t.s_base + v + ((long long)chunk << t.cb)
                          : t.s_base + (1LL << t.d0) - (1LL << t.cb) + v;
}

// ---------------------------------------------------------------------- top --
template <class E>
__global__ void __launch_bounds__(256) fx_top_kernel(const FxSeg* __restrict__ segs, int nseg,
                                                     const FxTree* __restrict__ trees,
                                                     const long long* __restrict__ lvl_off,
                                                     const double* __restrict__ roots, uint32_t* __restrict__ nodes,
                                                     typename fx_sum<E>::type* __restrict__ sval,
                                                     int* __restrict__ status) {
  typedef typename fx_sum<E>::type S;
  constexpr int L = sizeof(E) / 4;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ FxPivot<E> pv;
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  const FxSeg sg = segs[fx_find(segs, nseg, (long long)blockIdx.x)];
  const FxTree t = trees[sg.idx];
  const unsigned v = (unsigned)((long long)blockIdx.x - sg.first);  // (the top runs before any chunk: v' = v)
  const int d = 2 * t.n;
  E* C = reinterpret_cast<E*>(smem_raw);
  FxRow<E>* rows = reinterpret_cast<FxRow<E>*>(C + sym(d));
  S s = fx_of<S>(1.0);
  bool ok = true;
  for (int i = threadIdx.x; i < sym(d); i += blockDim.x) {
    const double x = roots[t.root_off + i];
    ok &= fx_root_entry_ok(x);
    C[i] = fx_of<E>(x);
  }
  __syncthreads();
  if (v == 0u && (int)threadIdx.x < t.n) {
    const int o = 2 * threadIdx.x;
    ok &= fx_root_mode_ok(C[tri(o, o)], C[tri(o + 1, o + 1)]);
  }
  for (unsigned left = v; left; left &= left - 1u) {
    const int o = 2 * (__ffs((int)left) - 1);
    if (threadIdx.x < 32) {  // one warp forms the pivot (every lane the same)
      FxPivot<E> q;
      ok &= fx_pivot(C[tri(o, o)], C[tri(o + 1, o)], C[tri(o + 1, o + 1)], q);
      s = umul(s, q.g);
      if (threadIdx.x == 0) pv = q;
    }
    __syncthreads();
    const int R = d - o - 2;
    for (int a = threadIdx.x; a < R; a += blockDim.x) fx_row(pv, C[tri(a + o + 2, o)], C[tri(a + o + 2, o + 1)], rows[a]);
    __syncthreads();
    for (int e = threadIdx.x; e < sym(R); e += blockDim.x) {
      int a = (int)((sqrtf(8.0f * (float)e + 1.0f) - 1.0f) * 0.5f);
      while (a * (a + 1) / 2 > e) --a;
      while ((a + 1) * (a + 2) / 2 <= e) ++a;
      const int b = e - a * (a + 1) / 2;
      E& c = C[tri(a + o + 2, b + o + 2)];
      c = fx_entry(c, rows[a].P, rows[a].Q, rows[a].A, rows[b].U, rows[b].V, rows[b].B);
    }
    __syncthreads();
  }
  int p;
  uint32_t* out;
  const bool tiled = v >= 32u;
  if (tiled) out = const_cast<uint32_t*>(fx_node<32, L>(nodes, lvl_off, t, v, 0u, p));
  else out = const_cast<uint32_t*>(fx_node<1, L>(nodes, lvl_off, t, v, 0u, p));
  const int o = d - 2 * p;
  for (int e = threadIdx.x; e < sym(2 * p); e += blockDim.x) {
    int a = (int)((sqrtf(8.0f * (float)e + 1.0f) - 1.0f) * 0.5f);
    while (a * (a + 1) / 2 > e) --a;
    while ((a + 1) * (a + 2) / 2 <= e) ++a;
    const int b = e - a * (a + 1) / 2;
    if (tiled) fx_st<E, 32>(out, e, C[tri(a + o, b + o)]); else fx_st<E, 1>(out, e, C[tri(a + o, b + o)]);
  }
  if (threadIdx.x == 0) sval[t.s_base + v] = s;
  if (!ok) atomicExch(status + t.tree, (int)kStatusRange);
}

// -------------------------------------------------------------------- level --
// Children of level k with q = R / 2 modes, when there are many: one warp per tile of
// 32, lane = child, no barrier.  Row a's P, Q, A are used at once, for entries (a, 0)
// .. (a, a); its U, V, B wait in shared memory for the rows below (2304 R bytes a warp
// with 6 limbs: 24 / 16 / 12 / 9 warps per SM at R = 4 / 6 / 8 / 10).  Bound by the
// multiply pipe at R = 4, 6 (70, 64 %, 4.4 TB/s beside it) and, with fewer warps, by
// the latency of its chains: NB entries at a time (FX, N = 24, q = 5, 4: 244, 278 us
// with 2, 213, 248 with 4, where 164 registers no longer cost warps; q = 3, 2: 312,
// 370 with 2, 328, 402 with 4), the next row's head loaded while this one is formed.
// Four warps sharing rows and entries behind barriers ran 683 us at q = 2 and 440 at q
// = 4 (one at a time: 371, 248).
template <class E, int ST, int NB>
__device__ __forceinline__ void fx_level_warp(const FxTree& t, const long long* lvl_off, int q, unsigned tile,
                                              unsigned chunk, uint32_t* nodes, typename fx_sum<E>::type* sval,
                                              int* status, uint32_t* sh) {
  constexpr int L = sizeof(E) / 4;
  const int lane = threadIdx.x & 31;
  const int R = 2 * q;
  const int k = t.n - 1 - q;
  const unsigned c = tile * 32u + lane;  // child of level k = parent node
  int p;
  const uint32_t* par = fx_node<ST, L>(nodes, lvl_off, t, c, chunk, p);
  const int o = 2 * (p - q - 1);  // the pivot's first row in the parent
  uint32_t* out = nodes + lvl_off[t.tab + k + 1] + (long long)tile * sym(R) * (L * 32) + lane;
  uint32_t* rowp = sh + lane;
  FxPivot<E> pv;
  const bool ok =
      fx_pivot(fx_ld<E, ST>(par, tri(o, o)), fx_ld<E, ST>(par, tri(o + 1, o)), fx_ld<E, ST>(par, tri(o + 1, o + 1)), pv);
  if (!ok) atomicExch(status + t.tree, (int)kStatusRange);
  sval[fx_sidx(t, (1u << (k - t.d0 + t.cb)) + c, chunk)] = umul(sval[fx_sidx(t, c, chunk)], pv.g);
  int e = 0;
  const uint32_t* src = par + (long long)tri(o + 2, o) * (L * ST);
  E u0 = fx_ld<E, ST>(src, 0), u1 = fx_ld<E, ST>(src, 1), cn = fx_ld<E, ST>(src, 2);
#pragma unroll 1
  for (int a = 0; a < R; ++a) {
    FxRow<E> r;
    fx_row(pv, u0, u1, r);
    E cc = cn;
    const uint32_t* next = src + (long long)(o + 3 + a) * (L * ST);  // row a + 1 is one entry longer
    if (a + 1 < R) {  // its head is on its way while this row's entries are formed
      u0 = fx_ld<E, ST>(next, 0);
      u1 = fx_ld<E, ST>(next, 1);
      cn = fx_ld<E, ST>(next, 2);
    }
    const uint32_t* x = rowp;
    int b = 0;
    // NB, then two entries at a time: their products' chains overlap
    if constexpr (NB == 4) {
#pragma unroll 1
      for (; b + 3 < a; b += 4, e += 4, x += 12 * L * 32) {
        const E c1 = fx_ld<E, ST>(src, b + 3), c2 = fx_ld<E, ST>(src, b + 4), c3 = fx_ld<E, ST>(src, b + 5);
        const E v0 = fx_entry(cc, r.P, r.Q, r.A, fx_ld<E, 32>(x, 0), fx_ld<E, 32>(x, 1), fx_ld<E, 32>(x, 2));
        cc = fx_ld<E, ST>(src, b + 6);
        const E v1 = fx_entry(c1, r.P, r.Q, r.A, fx_ld<E, 32>(x, 3), fx_ld<E, 32>(x, 4), fx_ld<E, 32>(x, 5));
        const E v2 = fx_entry(c2, r.P, r.Q, r.A, fx_ld<E, 32>(x, 6), fx_ld<E, 32>(x, 7), fx_ld<E, 32>(x, 8));
        const E v3 = fx_entry(c3, r.P, r.Q, r.A, fx_ld<E, 32>(x, 9), fx_ld<E, 32>(x, 10), fx_ld<E, 32>(x, 11));
        fx_st<E, 32>(out, e, v0);
        fx_st<E, 32>(out, e + 1, v1);
        fx_st<E, 32>(out, e + 2, v2);
        fx_st<E, 32>(out, e + 3, v3);
      }
    }
#pragma unroll 1
    for (; b + 1 < a; b += 2, e += 2, x += 6 * L * 32) {
      const E c1 = fx_ld<E, ST>(src, b + 3);
      const E v0 = fx_entry(cc, r.P, r.Q, r.A, fx_ld<E, 32>(x, 0), fx_ld<E, 32>(x, 1), fx_ld<E, 32>(x, 2));
      cc = fx_ld<E, ST>(src, b + 4);
      const E v1 = fx_entry(c1, r.P, r.Q, r.A, fx_ld<E, 32>(x, 3), fx_ld<E, 32>(x, 4), fx_ld<E, 32>(x, 5));
      fx_st<E, 32>(out, e, v0);
      fx_st<E, 32>(out, e + 1, v1);
    }
    if (b < a) {
      const E c1 = fx_ld<E, ST>(src, b + 3);
      fx_st<E, 32>(out, e, fx_entry(cc, r.P, r.Q, r.A, fx_ld<E, 32>(x, 0), fx_ld<E, 32>(x, 1), fx_ld<E, 32>(x, 2)));
      cc = c1;
      ++e;
    }
    fx_st<E, 32>(out, e, fx_entry(cc, r.P, r.Q, r.A, r.U, r.V, r.B));
    ++e;
    uint32_t* w = rowp + a * (3 * L * 32);
    fx_st<E, 32>(w, 0, r.U);
    fx_st<E, 32>(w, 1, r.V);
    fx_st<E, 32>(w, 2, r.B);
    src = next;
  }
}

template <class E, int NB>
__global__ void __launch_bounds__(32) fx_level_warp_kernel(const FxSeg* __restrict__ segs, int nseg,
                                                           const FxTree* __restrict__ trees,
                                                           const long long* __restrict__ lvl_off, int q, unsigned chunk,
                                                           uint32_t* nodes, typename fx_sum<E>::type* sval,
                                                           int* status) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const FxSeg sg = segs[fx_find(segs, nseg, (long long)blockIdx.x)];  // the plan is older than the top kernel
  const FxTree t = trees[sg.idx];
  fx_after();
  const unsigned tile = (unsigned)((long long)blockIdx.x - sg.first);
  // the first tile's parents are the root and levels 0 .. 4
  if (tile == 0u && chunk == 0u) fx_level_warp<E, 1, NB>(t, lvl_off, q, tile, chunk, nodes, sval, status, (uint32_t*)smem_raw);
  else fx_level_warp<E, 32, NB>(t, lvl_off, q, tile, chunk, nodes, sval, status, (uint32_t*)smem_raw);
}

// The same when children are few or their rows too many for that: a CTA takes TW (1 ..
// 16) consecutive children, and its 32 / TW x W lane groups share out the rows and then
// the entries.  One warp forms the pivots; the other CTAs of the SM hide it (q = 6, 7, 8
// at N = 24: 170, 108, 73 us with 16 children and 4 warps, 196, 123, 78 with 32 and 8).
// Spreading few children over the chip matters for the first levels: 32 .. 128 tiles
// of 32 took 42 - 54 us a level, now 14 - 24.
template <class E, int ST>
__device__ __forceinline__ void fx_level_cta(const FxTree& t, const long long* lvl_off, int q, unsigned c0, int TW,
                                             unsigned chunk, uint32_t* nodes, typename fx_sum<E>::type* sval,
                                             int* status, uint32_t* sh) {
  constexpr int L = sizeof(E) / 4;
  const int node = threadIdx.x & (TW - 1), worker = threadIdx.x / TW, workers = blockDim.x / TW;
  const int R = 2 * q;
  const int k = t.n - 1 - q;
  const unsigned c = c0 + node;
  int p;
  const uint32_t* par = fx_node<ST, L>(nodes, lvl_off, t, c, chunk, p);
  const int o = 2 * (p - q - 1);
  uint32_t* out = nodes + lvl_off[t.tab + k + 1] + (long long)(c >> 5) * sym(R) * (L * 32) + (c & 31u);
  // shared memory, word w of node i at w TW + i: the pivot's 5 values and flip, then 6
  // values per row (stride 6 L + 1 words, so that rows a group apart differ in bank)
  auto put = [&](uint32_t* w, const E& v) {
#pragma unroll
    for (int l = 0; l < L; ++l) w[l * TW] = v.w[l];
  };
  auto get = [&](const uint32_t* w) {
    E v;
#pragma unroll
    for (int l = 0; l < L; ++l) v.w[l] = w[l * TW];
    return v;
  };
  uint32_t* piv = sh + node;
  uint32_t* rowp = sh + (5 * L + 1) * TW + node;
  const int rs = (6 * L + 1) * TW, vs = L * TW;
  if (threadIdx.x < 32) {
    FxPivot<E> pv;
    const bool ok = fx_pivot(fx_ld<E, ST>(par, tri(o, o)), fx_ld<E, ST>(par, tri(o + 1, o)),
                             fx_ld<E, ST>(par, tri(o + 1, o + 1)), pv);
    if (worker == 0) {
      if (!ok) atomicExch(status + t.tree, (int)kStatusRange);
      sval[fx_sidx(t, (1u << (k - t.d0 + t.cb)) + c, chunk)] = umul(sval[fx_sidx(t, c, chunk)], pv.g);
      put(piv, pv.a);
      put(piv + vs, pv.b);
      put(piv + 2 * vs, pv.m);
      put(piv + 3 * vs, pv.c0);
      put(piv + 4 * vs, pv.c1);
      piv[5 * vs] = pv.flip;
    }
  }
  __syncthreads();
  {
    FxPivot<E> pv;
    pv.a = get(piv);
    pv.b = get(piv + vs);
    pv.m = get(piv + 2 * vs);
    pv.c0 = get(piv + 3 * vs);
    pv.c1 = get(piv + 4 * vs);
    pv.flip = piv[5 * vs];
#pragma unroll 1
    for (int a = worker; a < R; a += workers) {
      const int e = tri(o + 2 + a, o);
      FxRow<E> r;
      fx_row(pv, fx_ld<E, ST>(par, e), fx_ld<E, ST>(par, e + 1), r);
      uint32_t* w = rowp + a * rs;
      put(w, r.P);
      put(w + vs, r.Q);
      put(w + 2 * vs, r.A);
      put(w + 3 * vs, r.U);
      put(w + 4 * vs, r.V);
      put(w + 5 * vs, r.B);
    }
  }
  __syncthreads();
  const int ne = sym(R);
  int a = 0, b = worker;
#pragma unroll 1
  for (int e = worker; e < ne; e += workers, b += workers) {
    while (b > a) b -= ++a;
    const E cc = fx_ld<E, ST>(par, tri(o + 2 + a, o + 2) + b);
    const uint32_t *x = rowp + a * rs, *y = rowp + b * rs;
    fx_st<E, 32>(out, e, fx_entry(cc, get(x), get(x + vs), get(x + 2 * vs), get(y + 3 * vs), get(y + 4 * vs), get(y + 5 * vs)));
  }
}

template <class E>
__global__ void __launch_bounds__(256) fx_level_cta_kernel(const FxSeg* __restrict__ segs, int nseg,
                                                           const FxTree* __restrict__ trees,
                                                           const long long* __restrict__ lvl_off, int q, int TW,
                                                           unsigned chunk, uint32_t* nodes,
                                                           typename fx_sum<E>::type* sval, int* status) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const FxSeg sg = segs[fx_find(segs, nseg, (long long)blockIdx.x)];  // the plan is older than the top kernel
  const FxTree t = trees[sg.idx];
  fx_after();
  const unsigned c0 = (unsigned)((long long)blockIdx.x - sg.first) * (unsigned)TW;
  if (c0 < 32u && chunk == 0u) fx_level_cta<E, 1>(t, lvl_off, q, c0, TW, chunk, nodes, sval, status, (uint32_t*)smem_raw);
  else fx_level_cta<E, 32>(t, lvl_off, q, c0, TW, chunk, nodes, sval, status, (uint32_t*)smem_raw);
}

// --------------------------------------------------------------------- leaf --
// Sums of a thread: signed terms with (inc) and without (exc) the last mode, and all
// magnitudes.
template <class S>
struct FxSums {
  S inc, exc, mag;
};
// a + x, or a - x where mask is all ones (x ^ mask with the mask's carry).
template <int L, int F>
GBS_HD fxn<L, F> fx_add_signed(const fxn<L, F>& a, const fxn<L, F>& x, uint32_t mask) {
  fxn<L, F> t, r;
#pragma unroll
  for (int k = 0; k < L; ++k) t.w[k] = x.w[k] ^ mask;
  add_cc(mask, mask);  // carry = the mask's lowest bit
#pragma unroll
  for (int k = 0; k < L - 1; ++k) r.w[k] = addc_cc(a.w[k], t.w[k]);
  r.w[L - 1] = addc(a.w[L - 1], t.w[L - 1]);
  return r;
}

// The two subsets of a one-mode node: s g and s, of signs (-1)^neg and -(-1)^neg (neg
// all ones: odd).
template <class E, class S>
__device__ __forceinline__ bool fx_leaf1(const E& p00, const E& p10, const E& p11, const S& s, uint32_t neg,
                                         FxSums<S>& acc) {
  const E det = fx_det(p00, p10, p11);
  const S sg = umul(s, rsqrt_(det));
  acc.inc = fx_add_signed(acc.inc, sg, neg);
  acc.exc = fx_add_signed(acc.exc, s, ~neg);
  acc.mag = acc.mag + sg + s;
  return fx_det_in_range(det);
}

// The four subsets of the two-mode node in the four rows from o of a matrix.  Entries
// are read where they are used (the last block twice), which leaves registers for 16
// warps per SM.
template <class E, int ST, class S>
__device__ __forceinline__ bool fx_leaf2(const uint32_t* m, int o, const S& s, uint32_t neg, FxSums<S>& acc) {
  constexpr int W = sizeof(E) / 4 * ST;
  const uint32_t* m0 = m + (long long)tri(o, o) * W;
  const uint32_t* m1 = m + (long long)tri(o + 1, o) * W;
  const uint32_t* m2 = m + (long long)tri(o + 2, o) * W;
  const uint32_t* m3 = m + (long long)tri(o + 3, o) * W;
  FxPivot<E> pv;
  bool ok = fx_pivot(fx_ld<E, ST>(m0, 0), fx_ld<E, ST>(m1, 0), fx_ld<E, ST>(m1, 1), pv);
  FxRow<E> r;
  fx_row(pv, fx_ld<E, ST>(m2, 0), fx_ld<E, ST>(m2, 1), r);
  E p00 = fx_entry(fx_ld<E, ST>(m2, 2), r.P, r.Q, r.A, r.U, r.V, r.B);
  E p10, p11;
  {
    FxRow<E> r1;
    fx_row(pv, fx_ld<E, ST>(m3, 0), fx_ld<E, ST>(m3, 1), r1);
    p10 = fx_entry(fx_ld<E, ST>(m3, 2), r1.P, r1.Q, r1.A, r.U, r.V, r.B);
    p11 = fx_entry(fx_ld<E, ST>(m3, 3), r1.P, r1.Q, r1.A, r1.U, r1.V, r1.B);
  }
  S sv = umul(s, pv.g);
  // both sides through one copy of the code (the instruction cache is the limit of
  // an inlined one)
#pragma unroll 1
  for (int side = 0; side < 2; ++side) {
    ok &= fx_leaf1(p00, p10, p11, sv, neg ^ (0u - (uint32_t)side), acc);
    p00 = fx_ld<E, ST>(m2, 2);
    p10 = fx_ld<E, ST>(m3, 2);
    p11 = fx_ld<E, ST>(m3, 3);
    sv = s;
  }
  return ok;
}

template <class E, int Q, int ST>
__device__ __forceinline__ bool fx_leaf_node(const uint32_t* m, int p, const typename fx_sum<E>::type& s,
                                             uint32_t neg, FxSums<typename fx_sum<E>::type>& acc) {
  const int o = 2 * (p - Q);
  if constexpr (Q == 1) {
    return fx_leaf1(fx_ld<E, ST>(m, tri(o, o)), fx_ld<E, ST>(m, tri(o + 1, o)), fx_ld<E, ST>(m, tri(o + 1, o + 1)), s,
                    neg, acc);
  } else if constexpr (Q == 2) {
    return fx_leaf2<E, ST>(m, o, s, neg, acc);
  } else {
    // Three modes, for the narrow type (registers): the included child's ten entries are
    // formed row by row into local memory, the excluded one is a view.  356 us at N = 24
    // (64 fraction bits; 309 now) against 164 + 216 for a level launch that writes them and
    // a two-mode leaf that reads them back, and a launch less.
    static_assert(Q == 3, "at most three levels per leaf thread");
    constexpr int L = sizeof(E) / 4;
    uint32_t child[10 * L];
    typename fx_sum<E>::type sv;
    bool ok;
    {
      FxPivot<E> pv;
      ok = fx_pivot(fx_ld<E, ST>(m, tri(o, o)), fx_ld<E, ST>(m, tri(o + 1, o)), fx_ld<E, ST>(m, tri(o + 1, o + 1)), pv);
      sv = umul(s, pv.g);
      E U[4], V[4], B[4];
#pragma unroll
      for (int a = 0; a < 4; ++a) {
        const int e = tri(o + 2 + a, o);
        FxRow<E> r;
        fx_row(pv, fx_ld<E, ST>(m, e), fx_ld<E, ST>(m, e + 1), r);
        U[a] = r.U;
        V[a] = r.V;
        B[a] = r.B;
#pragma unroll
        for (int b = 0; b <= a; ++b)
          fx_st<E, 1>(child, tri(a, b), fx_entry(fx_ld<E, ST>(m, e + 2 + b), r.P, r.Q, r.A, U[b], V[b], B[b]));
      }
    }
    ok &= fx_leaf2<E, 1>(child, 0, sv, neg, acc);
    return fx_leaf2<E, ST>(m, o + 2, s, ~neg, acc) && ok;
  }
}

// Sum over a warp; every lane gets it.
template <class S>
__device__ __forceinline__ void fx_warp_sum(FxSums<S>& acc) {
#pragma unroll 1
  for (int off = 16; off > 0; off >>= 1) {
    acc.inc = acc.inc + shfl_xor(acc.inc, off);
    acc.exc = acc.exc + shfl_xor(acc.exc, off);
    acc.mag = acc.mag + shfl_xor(acc.mag, off);
  }
}

// A warp's tiles: every fourth of a unit's, from tile0 on.  Called behind the wait, so that what
// it reads does not change any more while it runs, and it may say so: without __restrict__ here
// the loads are ordered worse and spill (N = 24, 64, 128, 160 bits: 334, 428, 560 us, 310, 410,
// 536 with it).
template <class E, int Q>
__device__ __forceinline__ bool fx_leaf_tiles(const FxTree& t, const long long* __restrict__ lvl_off,
                                              const uint32_t* __restrict__ nodes,
                                              const typename fx_sum<E>::type* __restrict__ sval, unsigned tile0, int tiles,
                                              unsigned chunk, FxSums<typename fx_sum<E>::type>& acc) {
  typedef typename fx_sum<E>::type S;
  constexpr int L = sizeof(E) / 4;
  const int lane = threadIdx.x & 31;
  const unsigned count = 1u << (t.D - t.d0 + t.cb);
  bool ok = true;
#pragma unroll 1
  for (int i = 0; i < tiles; ++i) {
    const unsigned v = (tile0 + 4u * i) * 32u + lane;
    if (v >= count) break;
    const S s = sval[fx_sidx(t, v, chunk)];
    // sign of the node: (-1)^(exclusions above)
    const uint32_t odd = ((t.D - __popc(v) - __popc(chunk)) & 1) ? 0xffffffffu : 0u;
    int p;
    if (v < 32u && chunk == 0u) {
      const uint32_t* m = fx_node<1, L>(nodes, lvl_off, t, v, chunk, p);
      ok &= fx_leaf_node<E, Q, 1>(m, p, s, odd, acc);
    } else {
      const uint32_t* m = fx_node<32, L>(nodes, lvl_off, t, v, chunk, p);
      ok &= fx_leaf_node<E, Q, 32>(m, p, s, odd, acc);
    }
  }
  return ok;
}

// One CTA of four warps per unit: 4 x tiles_per_unit consecutive tiles of 32 nodes of one
// tree, one partial sum.
template <class E, int Q>
__global__ void __launch_bounds__(128, 4) fx_leaf_kernel(const FxSeg* __restrict__ segs, int nseg, unsigned chunk,
                                                         const FxTree* __restrict__ trees,
                                                         const long long* __restrict__ lvl_off,
                                                         const uint32_t* nodes,
                                                         const typename fx_sum<E>::type* sval,
                                                         FxPart<typename fx_sum<E>::type>* parts,
                                                         int* status) {
  typedef typename fx_sum<E>::type S;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const FxSeg sg = segs[fx_find(segs, nseg, (long long)blockIdx.x)];  // the plan is older than the top kernel
  const FxTree t = trees[sg.idx];
  fx_after();
  const S zero = fx_of<S>(0.0);
  FxSums<S> acc{zero, zero, zero};
  const unsigned tile0 = (unsigned)((long long)blockIdx.x - sg.first) * 4u * (unsigned)sg.tiles_per_unit + warp;
  const bool ok = fx_leaf_tiles<E, Q>(t, lvl_off, nodes, sval, tile0, sg.tiles_per_unit, chunk, acc);
  if (!ok) atomicExch(status + t.tree, (int)kStatusRange);
  __syncwarp();
  fx_warp_sum(acc);
  __shared__ FxPart<S> sh[4];
  if (lane == 0) sh[warp] = FxPart<S>{acc.inc, acc.exc, acc.mag};
  __syncthreads();
  if (threadIdx.x == 0) {
    for (int w = 1; w < 4; ++w) {
      acc.inc = acc.inc + sh[w].inc;
      acc.exc = acc.exc + sh[w].exc;
      acc.mag = acc.mag + sh[w].abs;
    }
    parts[blockIdx.x] = FxPart<S>{acc.inc, acc.exc, acc.mag};
  }
}

// -------------------------------------------------------------------- final --
// One CTA per tree; segs[t].first = the tree's first unit, segs[t + 1].first the end.
// (Ten thousand partial sums took it 31 us; a sum per leaf CTA leaves it some thousand.)
template <class S>
__global__ void __launch_bounds__(1024) fx_final_kernel(const FxPart<S>* parts,
                                                        const FxSeg* __restrict__ segs,
                                                        const FxTree* __restrict__ trees,
                                                        const int* status, double u, double extra,
                                                        ProbOut* out) {
  fx_after();
  const int t = blockIdx.x;
  const S zero = fx_of<S>(0.0);
  S inc = zero, exc = zero, mag = zero;
  for (long long i = segs[t].first + threadIdx.x; i < segs[t + 1].first; i += blockDim.x) {
    inc = inc + parts[i].inc;
    exc = exc + parts[i].exc;
    mag = mag + parts[i].abs;
  }
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
  __shared__ FxPart<S> sh[32];
#pragma unroll 1
  for (int stage = 0; stage < 2; ++stage) {
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) {
      inc = inc + shfl_down(inc, off);
      exc = exc + shfl_down(exc, off);
      mag = mag + shfl_down(mag, off);
    }
    if (stage == 1) break;
    if (lane == 0) sh[warp] = FxPart<S>{inc, exc, mag};
    __syncthreads();
    if (warp != 0) return;
    inc = lane < nw ? sh[lane].inc : zero;
    exc = lane < nw ? sh[lane].exc : zero;
    mag = lane < nw ? sh[lane].abs : zero;
  }
  if (lane != 0) return;
  const FxTree tr = trees[segs[t].idx];
  TreeOut o;
  fx_store3(inc, o.inc);
  fx_store3(exc, o.exc);
  o.abs = to_double(mag);
  out[tr.tree] = finish_tree(o, status[tr.tree], tr.scale, tr.n, u, extra);
}

// -------------------------------------------------------------- small trees --
// A tree of few modes is latency only, so it takes one launch.  A CTA per setting of
// the tree's first d0 modes (none for the smallest): it eliminates the included ones
// from the root in shared memory, and then grows the remaining nsub modes' tree there,
// breadth first.  A level takes two phases shared out among all threads: the rows, then
// the entries together with the next level's pivots (a child's three pivot entries are
// formed twice, which takes the pivots' long chain off the path).  Two threads per node
// with two modes left form its four terms.  The last CTA of a tree to finish adds the
// CTAs' sums (exact integers: in any order) and finishes the result.
struct FxSmall {
  long long first;  // first CTA (and partial sum) of this tree
  long long root_off;
  double scale;  // det(Sigma)^(-1/2)
  int n, d0, tree, pad;
};

// A row in shared memory, an odd number of words long (6 L is even).
template <class E>
struct FxRowPad : FxRow<E> {
  uint32_t pad;
};

// Shared memory in words: root, the nsub-mode tree's levels, s of its nodes, pivots and
// rows of the widest level.
__host__ __device__ constexpr int fx_small_words(int n, int nsub, int L, int LS) {
  const int D = nsub > 2 ? nsub - 2 : 0;
  int words = sym(2 * n) * L + (1 << D) * LS, rows = nsub < n ? 2 * n : 0;
  for (int k = 0; k < D; ++k) {
    words += (1 << k) * sym(2 * (nsub - 1 - k)) * L;
    const int r = (1 << k) * 2 * (nsub - 1 - k);
    rows = r > rows ? r : rows;
  }
  return words + (D > 0 ? (1 << (D - 1)) : 1) * (6 * L + 1) + rows * (6 * L + 1);
}

// The operations on values in memory, inlined (CALL = false) or as functions of their
// own.  A kernel that holds one type's tree inlines them; one that holds four (the
// sampler's chain) calls them, or the instruction caches thrash: graph sampling of 100
// modes 45 ms with calls, 53 without; a tree of 9 modes alone (128 fraction bits) 33 us
// with, 27 without.
template <class E>
__device__ __forceinline__ bool fxm_pivot(const E* p00, const E* p10, const E* p11, FxPivot<E>* pv) {
  FxPivot<E> r;
  const bool ok = fx_pivot(*p00, *p10, *p11, r);
  *pv = r;
  return ok;
}
template <class E>
__device__ __forceinline__ void fxm_row(const FxPivot<E>* pv, const E* u0, const E* u1, FxRow<E>* out) {
  FxRow<E> r;
  fx_row(*pv, *u0, *u1, r);
  *out = r;
}
template <class E>
__device__ __forceinline__ void fxm_entry(const E* c, const FxRow<E>* a, const FxRow<E>* b, E* out) {
  *out = fx_entry(*c, a->P, a->Q, a->A, b->U, b->V, b->B);
}
// The pivot block of a child, entries (0, 0), (1, 0), (1, 1): c and d are the parent's
// (0, 0) and (1, 0).  Together, so that their chains overlap.
template <class E>
__device__ __forceinline__ void fxm_block(const E* c, const E* d, const FxRowPad<E>* r, E* out) {
  const E x = fx_entry(*c, r[0].P, r[0].Q, r[0].A, r[0].U, r[0].V, r[0].B);
  const E y = fx_entry(d[0], r[1].P, r[1].Q, r[1].A, r[0].U, r[0].V, r[0].B);
  const E z = fx_entry(d[1], r[1].P, r[1].Q, r[1].A, r[1].U, r[1].V, r[1].B);
  out[0] = x;
  out[1] = y;
  out[2] = z;
}
template <class E, class S>
__device__ __forceinline__ bool fxm_leaf1(const E* p00, const E* p10, const E* p11, const S* s, uint32_t neg,
                                          FxSums<S>* acc) {
  FxSums<S> t = *acc;
  const bool ok = fx_leaf1(*p00, *p10, *p11, *s, neg, t);
  *acc = t;
  return ok;
}
template <class E>
__device__ __noinline__ bool fxc_pivot(const E* p00, const E* p10, const E* p11, FxPivot<E>* pv) {
  return fxm_pivot(p00, p10, p11, pv);
}
template <class E>
__device__ __noinline__ void fxc_row(const FxPivot<E>* pv, const E* u0, const E* u1, FxRow<E>* out) {
  fxm_row(pv, u0, u1, out);
}
template <class E>
__device__ __noinline__ void fxc_entry(const E* c, const FxRow<E>* a, const FxRow<E>* b, E* out) {
  fxm_entry(c, a, b, out);
}
template <class E>
__device__ __noinline__ void fxc_block(const E* c, const E* d, const FxRowPad<E>* r, E* out) {
  fxm_block(c, d, r, out);
}
template <class E, class S>
__device__ __noinline__ bool fxc_leaf1(const E* p00, const E* p10, const E* p11, const S* s, uint32_t neg,
                                       FxSums<S>* acc) {
  return fxm_leaf1(p00, p10, p11, s, neg, acc);
}
template <class E, bool CALL>
struct FxOps {
  typedef typename fx_sum<E>::type S;
  static __device__ __forceinline__ bool pivot(const E* p00, const E* p10, const E* p11, FxPivot<E>* pv) {
    if constexpr (CALL) return fxc_pivot(p00, p10, p11, pv); else return fxm_pivot(p00, p10, p11, pv);
  }
  static __device__ __forceinline__ void row(const FxPivot<E>* pv, const E* u0, const E* u1, FxRow<E>* out) {
    if constexpr (CALL) fxc_row(pv, u0, u1, out); else fxm_row(pv, u0, u1, out);
  }
  static __device__ __forceinline__ void entry(const E* c, const FxRow<E>* a, const FxRow<E>* b, E* out) {
    if constexpr (CALL) fxc_entry(c, a, b, out); else fxm_entry(c, a, b, out);
  }
  static __device__ __forceinline__ void block(const E* c, const E* d, const FxRowPad<E>* r, E* out) {
    if constexpr (CALL) fxc_block(c, d, r, out); else fxm_block(c, d, r, out);
  }
  static __device__ __forceinline__ bool leaf1(const E* p00, const E* p10, const E* p11, const S* s, uint32_t neg,
                                               FxSums<S>* acc) {
    if constexpr (CALL) return fxc_leaf1(p00, p10, p11, s, neg, acc); else return fxm_leaf1(p00, p10, p11, s, neg, acc);
  }
};

// The tree of a CTA: the n-mode root (root(i): entry i of its packed triangle) with the
// first d0 modes set to pre, all other subsets enumerated.  Returns the CTA's sums in
// its first warp (every lane); ok turns false in the threads that met a pivot out of
// range.  Ends without a barrier: one is needed before smem is used again.
template <class E, bool CALL, class Root>
__device__ __forceinline__ FxPart<typename fx_sum<E>::type> fx_cta_tree(unsigned char* smem, int n, int d0, unsigned pre,
                                                                        const Root& root, bool& ok) {
  typedef typename fx_sum<E>::type S;
  typedef FxOps<E, CALL> Op;
  const int ns = n - d0, D = ns > 2 ? ns - 2 : 0, nthr = blockDim.x;
  E* mats = reinterpret_cast<E*>(smem);
  __shared__ int lvl[16];           // entries before level k (the root first)
  __shared__ uint16_t tab[595];     // packed entry -> (row, column), sym(34) of them
  __shared__ int base[256];         // node -> first entry of its matrix
  __shared__ unsigned char held[256];  // node -> modes of its matrix
  if (threadIdx.x == 0) {
    int o = sym(2 * n);
    for (int k = 0; k <= D; ++k) {
      lvl[k] = o;
      o += (1 << k) * sym(2 * (ns - 1 - k));
    }
  }
  for (int i = threadIdx.x; i < sym(2 * n); i += nthr) {
    const double x = root(i);
    ok &= fx_root_entry_ok(x);
    mats[i] = fx_of<E>(x);
    int a = (int)((sqrtf(8.0f * (float)i + 1.0f) - 1.0f) * 0.5f);
    while (a * (a + 1) / 2 > i) --a;
    while ((a + 1) * (a + 2) / 2 <= i) ++a;
    tab[i] = (uint16_t)(a << 8 | (i - a * (a + 1) / 2));
  }
  __syncthreads();
  for (int v = threadIdx.x; v < (1 << D); v += nthr) {
    const int k = 31 - __clz(v | 1), p = v ? ns - 1 - k : n;
    base[v] = v ? lvl[k] + (v - (1 << k)) * sym(2 * p) : 0;
    held[v] = (unsigned char)p;
  }
  if ((int)threadIdx.x < n) {
    const int o = 2 * threadIdx.x;
    ok &= fx_root_mode_ok(mats[tri(o, o)], mats[tri(o + 1, o + 1)]);
  }
  S* sv = reinterpret_cast<S*>(mats + lvl[D]);
  FxPivot<E>* piv = reinterpret_cast<FxPivot<E>*>(sv + (1 << D));
  FxRowPad<E>* rows = reinterpret_cast<FxRowPad<E>*>(piv + (D > 0 ? 1 << (D - 1) : 1));
  // ---- the included modes among the first d0
  if (threadIdx.x == 0) sv[0] = fx_of<S>(1.0);
  for (unsigned left = pre; left; left &= left - 1u) {
    const int o = 2 * (__ffs((int)left) - 1), R = 2 * n - o - 2;
    if (threadIdx.x == 0) {
      ok &= Op::pivot(mats + tri(o, o), mats + tri(o + 1, o), mats + tri(o + 1, o + 1), piv);
      sv[0] = umul(sv[0], piv[0].g);
    }
    __syncthreads();
    for (int a = threadIdx.x; a < R; a += nthr) {
      const E* m = mats + tri(a + o + 2, o);
      Op::row(piv, m, m + 1, rows + a);
    }
    __syncthreads();
    for (int e = threadIdx.x; e < sym(R); e += nthr) {
      const int a = tab[e] >> 8, b = tab[e] & 255;
      E* c = mats + tri(a + o + 2, b + o + 2);
      Op::entry(c, rows + a, rows + b, c);
    }
    __syncthreads();
  }
  // ---- the tree of the other ns modes: node v's matrix, and the first row of its
  // view with q modes
  auto node = [&](int v, int q, int& o) {
    o = 2 * ((int)held[v] - q);
    return mats + base[v];
  };
  // level -1: the pivot of node 0; level k: its rows, then its entries together with the
  // pivots of nodes 0 .. 2^(k+1) - 1 at depth k + 1, by the first threads, which form the
  // pivot entries of the new ones themselves
  for (int k = -1; k < D; ++k) {
    const int q = ns - 1 - k, R = 2 * q, nc = k < 0 ? 0 : 1 << k;
    const float inv_r = 1.0f / (float)R;
    for (int i = threadIdx.x; i < nc * R; i += nthr) {
      const int c = (int)(((float)i + 0.5f) * inv_r), a = i - c * R;  // exact: i < 2^10
      int o;
      const E* m = node(c, q + 1, o) + tri(o + 2 + a, o);
      Op::row(piv + c, m, m + 1, rows + i);
    }
    __syncthreads();
    const int np = k + 1 < D ? max(2 * nc, 1) : 0, ne = sym(R);
    const int skip = min((np + 31) & ~31, nthr / 2);
    const float inv_e = 1.0f / (float)ne;
    E* dst = mats + lvl[max(k, 0)];
    auto entry = [&](int c, int e) {
      const int ab = tab[e], a = ab >> 8, b = ab & 255;
      int o;
      const E* m = node(c, q + 1, o);
      Op::entry(m + tri(o + 2 + a, o + 2) + b, rows + c * R + a, rows + c * R + b, dst + c * ne + e);
    };
    // entries e >= first of a child are the other threads'
    const int first = np ? 3 : 0, per = ne - first;
    const float inv_p = 1.0f / (float)per;
    const bool pivots = (int)threadIdx.x < skip;
    for (int v = pivots || np > skip ? threadIdx.x : np; v < np; v += nthr) {
      int o = 0;
      const E* m;
      if (v < nc || k < 0) {
        m = node(v, q, o);
      } else {
        const E* par = node(v - nc, q + 1, o);
        Op::block(par + tri(o + 2, o + 2), par + tri(o + 3, o + 2), rows + (v - nc) * R, dst + (v - nc) * ne);
        o = 0;
        m = dst + (v - nc) * ne;
      }
      ok &= Op::pivot(m + tri(o, o), m + tri(o + 1, o), m + tri(o + 1, o + 1), piv + v);
      sv[max(2 * nc, 1) + v] = umul(sv[v], piv[v].g);
    }
    if (!pivots) {
      for (int i = threadIdx.x - skip; i < nc * per; i += nthr - skip) {
        const int c = (int)(((float)i + 0.5f) * inv_p);  // exact: i < 2^11
        entry(c, i - c * per + first);
      }
    }
    __syncthreads();
  }
  const S zero = fx_of<S>(0.0);
  FxSums<S> acc{zero, zero, zero};
  const int above = n - (ns < 2 ? 1 : 2) - __popc(pre);  // decided modes but the prefix's included ones
  if (ns == 1) {
    if (threadIdx.x == 0) {
      int o;
      const E* m = node(0, 1, o);
      ok &= Op::leaf1(m + tri(o, o), m + tri(o + 1, o), m + tri(o + 1, o + 1), sv, (above & 1) ? 0xffffffffu : 0u, &acc);
    }
  } else {
    // two threads per two-mode node: the subsets with its first mode, and those without
    for (int i = threadIdx.x; i < (2 << D); i += nthr) {
      const int v = i & ((1 << D) - 1), side = i >> D;
      const uint32_t neg = ((above - __popc(v) - side) & 1) ? 0xffffffffu : 0u;
      int o;
      const E* m = node(v, 2, o);
      const E *m2 = m + tri(o + 2, o), *m3 = m + tri(o + 3, o);
      const E *p00 = m2 + 2, *p10 = m3 + 2, *p11 = m3 + 3;
      const S* s = sv + v;
      E p[3];
      S sg;
      if (side == 0) {
        FxPivot<E> pv;
        FxRow<E> r0, r1;
        ok &= Op::pivot(m + tri(o, o), m + tri(o + 1, o), m + tri(o + 1, o + 1), &pv);
        Op::row(&pv, m2, m2 + 1, &r0);
        Op::row(&pv, m3, m3 + 1, &r1);
        Op::entry(p00, &r0, &r0, p);
        Op::entry(p10, &r1, &r0, p + 1);
        Op::entry(p11, &r1, &r1, p + 2);
        sg = umul(*s, pv.g);
        p00 = p;
        p10 = p + 1;
        p11 = p + 2;
        s = &sg;
      }
      ok &= Op::leaf1(p00, p10, p11, s, neg, &acc);
    }
  }
  __shared__ FxPart<S> sh[16];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  fx_warp_sum(acc);
  if (lane == 0) sh[warp] = FxPart<S>{acc.inc, acc.exc, acc.mag};
  __syncthreads();
  if (warp == 0) {
    const int nw = nthr >> 5;
    acc.inc = lane < nw ? sh[lane].inc : zero;
    acc.exc = lane < nw ? sh[lane].exc : zero;
    acc.mag = lane < nw ? sh[lane].abs : zero;
    fx_warp_sum(acc);
  }
  return FxPart<S>{acc.inc, acc.exc, acc.mag};
}

template <class E>
__global__ void __launch_bounds__(512) fx_small_kernel(const FxSmall* __restrict__ trees, int ntrees,
                                                       const double* __restrict__ roots, double u, double extra,
                                                       FxPart<typename fx_sum<E>::type>* __restrict__ parts,
                                                       int* __restrict__ counts, int* __restrict__ status,
                                                       ProbOut* __restrict__ out) {
  typedef typename fx_sum<E>::type S;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ int last, bad;
  int lo = 0, hi = ntrees - 1;
  while (lo < hi) {
    const int mid = (lo + hi + 1) >> 1;
    if (trees[mid].first <= (long long)blockIdx.x) lo = mid; else hi = mid - 1;
  }
  const FxSmall t = trees[lo];
  const unsigned pre = (unsigned)((long long)blockIdx.x - t.first);
  bool ok = true;
  if (threadIdx.x == 0) bad = 0;
  FxPart<S> sum = fx_cta_tree<E, false>(smem_raw, t.n, t.d0, pre, [&](int i) { return roots[t.root_off + i]; }, ok);
  if (!ok) bad = 1;
  __syncthreads();
  const int lane = threadIdx.x & 31;
  if (threadIdx.x >= 32) return;
  int st = bad ? (int)kStatusRange : (int)kStatusOk;
  if (t.d0 > 0) {
    if (lane == 0) {
      if (bad) atomicExch(status + t.tree, (int)kStatusRange);
      parts[blockIdx.x] = sum;
      __threadfence();
      last = atomicAdd(counts + t.tree, 1) == (1 << t.d0) - 1;
    }
    __syncwarp();
    if (!last) return;
    __threadfence();
    const S zero = fx_of<S>(0.0);
    FxSums<S> acc{zero, zero, zero};
    for (int i = lane; i < (1 << t.d0); i += 32) {
      const volatile uint32_t* w = reinterpret_cast<const volatile uint32_t*>(parts + t.first + i);
      FxPart<S> q;
#pragma unroll
      for (int k = 0; k < (int)(sizeof(S) / 4); ++k) {
        q.inc.w[k] = w[k];
        q.exc.w[k] = w[sizeof(S) / 4 + k];
        q.abs.w[k] = w[2 * (sizeof(S) / 4) + k];
      }
      acc.inc = acc.inc + q.inc;
      acc.exc = acc.exc + q.exc;
      acc.mag = acc.mag + q.abs;
    }
    fx_warp_sum(acc);
    sum = FxPart<S>{acc.inc, acc.exc, acc.mag};
    st = *(volatile int*)(status + t.tree);
  }
  if (lane != 0) return;
  TreeOut o;
  fx_store3(sum.inc, o.inc);
  fx_store3(sum.exc, o.exc);
  o.abs = to_double(sum.abs);
  out[t.tree] = finish_tree(o, st, t.scale, t.n, u, extra);
}

}  // namespace gbs
