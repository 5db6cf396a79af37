// Batched probabilities: staging arena, batched click blocks, per-tree finish,
// the precision ladder over a batch, and gbs_torontonian_batch.
#include <algorithm>
#include <cmath>
#include <cstdio>
#include <cstring>
#include <string>
#include <vector>

#include "gbs_batch_driver.cuh"
#include "gbs_internal.h"

namespace gbs {

gbs_status stage_begin(gbs_ctx* ctx, size_t bytes) {
  bytes = (bytes + 4096 + 255) / 256 * 256;
  StageArena& a = ctx->stage;
  gbs_status st;
  if (bytes > a.cap) {
    if ((st = stream_sync(ctx))) return st;
    size_t cap = std::max(bytes, a.cap * 2);
    cap = std::max(cap, (size_t)1 << 20);
    if (ctx->stage_host) cudaFreeHost(ctx->stage_host);
    ctx->stage_host = nullptr;
    a.cap = 0;
    if ((st = check_cuda(ctx, cudaMallocHost(&ctx->stage_host, cap), "pinned staging"))) return st;
    dev_free(ctx, ctx->stage_dev);
    if ((st = dev_alloc(ctx, ctx->stage_dev, cap))) return st;
    a.cap = cap;
  }
  if (a.begin()) {
    if ((st = stream_sync(ctx))) return st;
    a.begin();
  }
  return GBS_OK;
}

gbs_status stage(gbs_ctx* ctx, const void* data, size_t bytes, const void** dev) {
  StageArena& a = ctx->stage;
  if (!a.fits(bytes)) return set_error(ctx, GBS_ENOMEM, "staging arena too small for this call");
  gbs_status st;
  if (!a.clear(bytes) && (st = stream_sync(ctx))) return st;
  const size_t off = a.take(bytes);
  unsigned char* h = (unsigned char*)ctx->stage_host + off;
  unsigned char* d = (unsigned char*)ctx->stage_dev.ptr + off;
  *dev = d;
  if (!bytes) return GBS_OK;
  memcpy(h, data, bytes);
  return check_cuda(ctx, cudaMemcpyAsync(d, h, bytes, cudaMemcpyHostToDevice, ctx->stream), "stage copy");
}

const BatchTune& batch_tune_for(gbs_ctx* ctx, int prec, bool real) {
  return ctx->tune[prec < 0 || prec > kTuneLast ? 1 : prec][real ? 1 : 0];
}

// Every value of a tree over n modes of (Sigma^-1)_S fits the fixed-point range: its
// eigenvalues are at least 1/sigma_max, which bounds the scaled pivot inverses by
// sigma_max, each included pivot's factor of s by sigma_max and the sums by
// (1 + sigma_max)^n (inside the 63-bit integer part of s and the sums).  Entries and pivot
// determinants are bounded where Sigma >= I/2 (a physical state: 2 and 4); a covariance
// given as such promises Sigma > 0 only, so the engine checks the root itself.
bool fx_ok_inverse(const gbs_state* st, int n) {
  const double sm = st->sigma_max;
  return sm > 0.0 && sm <= 1024.0 && n * std::log2(1.0 + sm) < 60.0;
}
// A tree over a conditioned Sigma' (sampler): Sigma' >= I/2 bounds the pivot
// determinants below by 1/4, so s <= 2^n and the sums <= 3^n; entries and
// determinants are bounded by sigma_max and sigma_max^2.
bool fx_ok_sigma(const gbs_state* st, int n) {
  const double sm = st->sigma_max;
  return sm > 0.0 && sm < 64.0 && n <= 36;
}

// FP64 trees in 64-bit fixed point (64 fraction bits; s and sums have 95 integer bits).
// A Schur step rounds an entry by up to 2^-60 of what it takes off it (the inverse square
// root's 2^-61, squared) and some products' 2^-64 each, all low; FP64 by 2^-53 of the entry
// and of what is taken off it.  Whatever either leaves goes through the same later steps: a
// factor of up to 1 + |L|^2 <= 1 + 2 sigma_max in an entry, and of 2 sigma_max from an entry
// to a relative determinant.  With sigma_max <= 16 entries lie in [1/16, 2] on the diagonal, so
// a step here rounds by less than 2^-59 where FP64 rounds by 2^-57 at least, and the tree keeps
// FP64's error estimate.  (That estimate, 4 n + 24 units per term, is a model for either: the
// worst case over all steps, n^2 2^-59 (1 + 2 sigma_max) sigma_max relative, would pass it 30-fold
// at sigma_max = 16, n = 22, and FP64's by more.  Measured there, n = 4 .. 22: at most 4e-4 of
// the estimate, 0.13 in FP64; 5e-5 and 0.06 at sigma_max = 8.)
// Every term of a physical state's (Sigma^-1)_S tree is at least 1 (det of a conditioned V +
// I/2 is), so the sum of magnitudes is at least 2^n and the terms' absolute errors vanish
// against FP64's.  The bound needs the closed form (a state built from its factors).
bool fxd_ok_inverse(const gbs_state* st, int n) {
  const double sm = st->sigma_max;
  return st->has_factors && sm > 0.0 && sm <= 16.0 && n * std::log2(1.0 + sm) < 92.0;
}
// Sampler trees: entries up to 64, rounded relative to what a step takes off them as above.
// Terms are at most 1, and their magnitudes add up to at least 1; a term's s is a product of
// factors in [1/64, 2], truncated to 2^-64 at each, so 2^10 terms of 10 factors are off by less
// than 2^-50 together, against an estimate of 64 2^-53 of the sum of magnitudes at least.
bool fxd_ok_sigma(const gbs_state* st, int n) { return fx_ok_sigma(st, n) && n <= 10; }

// ------------------------------------------------------- click blocks ---
struct ClickReq {
  const cplx<double>* U;      // factor form (or null)
  const double* alpha;
  const double* beta;
  const cplx<double>* Sinv;   // dense form (when U is null)
  long long root_off;
  int M, N;
  ModeList S;
};

// The 2 x 2 block of (Sigma^-1) between two modes: [[h00, h01], [h10, h11]] in (a, a^+).
struct ClickEntry {
  cplx<double> h00, h01, h10, h11;
};
__device__ __forceinline__ ClickEntry click_entry_dense(const ClickReq& q, int j, int k) {
  const long long M = q.M, D = 2 * M;
  const long long rj = q.S.m[j], rk = q.S.m[k];
  return ClickEntry{q.Sinv[rj * D + rk], q.Sinv[rj * D + rk + M], q.Sinv[(rj + M) * D + rk], q.Sinv[(rj + M) * D + rk + M]};
}
// Writes the block of mode pair (j, k) into the request's packed root.
__device__ __forceinline__ void click_store(const ClickReq& q, int j, int k, ClickEntry h, int real_basis,
                                            void* __restrict__ roots) {
  if (j == k) h.h00.im = h.h11.im = 0.0;
  const int a0 = 2 * j, b0 = 2 * k;
  auto T3 = [](int a, int b) { return a * (a + 1) / 2 + b; };
  if (real_basis) {
    // q^+ h q with q = [[1, i], [1, -i]]/sqrt2
    double* o = (double*)roots + q.root_off;
    o[T3(a0, b0)] = 0.5 * (h.h00.re + h.h01.re + h.h10.re + h.h11.re);
    o[T3(a0 + 1, b0)] = 0.5 * ((h.h00.im + h.h01.im) - (h.h10.im + h.h11.im));
    o[T3(a0 + 1, b0 + 1)] = 0.5 * ((h.h00.re - h.h01.re) - (h.h10.re - h.h11.re));
    if (j != k) o[T3(a0, b0 + 1)] = -0.5 * (h.h00.im - h.h01.im + h.h10.im - h.h11.im);
  } else {
    cplx<double>* o = (cplx<double>*)roots + q.root_off;
    o[T3(a0, b0)] = h.h00;
    o[T3(a0 + 1, b0)] = h.h10;
    o[T3(a0 + 1, b0 + 1)] = h.h11;
    if (j != k) o[T3(a0, b0 + 1)] = h.h01;
  }
}

// Mode pair (j, k) of index p in the packed triangle.
__device__ __forceinline__ void click_pair(int p, int* j, int* k) {
  int r = (int)((sqrtf(8.0f * (float)p + 1.0f) - 1.0f) * 0.5f);
  while (r * (r + 1) / 2 > p) --r;
  while ((r + 1) * (r + 2) / 2 <= p) ++r;
  *j = r;
  *k = p - r * (r + 1) / 2;
}
// The sums over l of A = (Sigma^-1)_{a_j a_k}, B = (Sigma^-1)_{a_j a^+_k}: runs of kClickL
// in kClickS strided parts of 8, the parts summed over the runs and joined in pairs.  Both
// kernels below add the same numbers in this order, so a request's root does not depend
// on its batch; its rounding is that of a sum over 32 lanes.
constexpr int kClickS = 4, kClickL = 32;
struct ClickSum {
  double ar = 0, ai = 0, br = 0, bi = 0;
  __device__ __forceinline__ void step(cplx<double> x, cplx<double> v, double alpha, double beta) {
    const double rr = x.re * v.re, ri = x.re * v.im;
    ar = fma(fma(x.im, v.im, rr), alpha, ar);
    ai = fma(fma(x.im, v.re, -ri), alpha, ai);
    br = fma(fma(-x.im, v.im, rr), beta, br);
    bi = fma(fma(x.im, v.re, ri), beta, bi);
  }
  __device__ __forceinline__ void add(const ClickSum& o) {
    ar += o.ar;
    ai += o.ai;
    br += o.br;
    bi += o.bi;
  }
  // lane i's of each 16 lanes
  __device__ __forceinline__ ClickSum from(int i) const {
    return ClickSum{__shfl_sync(0xffffffffu, ar, i, 16), __shfl_sync(0xffffffffu, ai, i, 16),
                    __shfl_sync(0xffffffffu, br, i, 16), __shfl_sync(0xffffffffu, bi, i, 16)};
  }
  __device__ __forceinline__ ClickEntry entry() const { return ClickEntry{{ar, ai}, {br, bi}, {br, -bi}, {ar, -ai}}; }
};

// Few requests: kClickG groups of kClickS lanes per (request, mode pair j >= k), a run a
// group, blockIdx.x the request; writes the packed lower triangle.  Bound by the latency
// of the loads, which a lane issues together.
constexpr int kClickG = 4, kClickPair = kClickG * kClickS;
__global__ void __launch_bounds__(128) batch_click_block_kernel(const ClickReq* __restrict__ reqs, int real_basis,
                                                                void* __restrict__ roots) {
  __shared__ ClickReq q;
  for (int i = threadIdx.x; i < (int)(sizeof(ClickReq) / 4); i += blockDim.x)
    reinterpret_cast<int*>(&q)[i] = reinterpret_cast<const int*>(reqs + blockIdx.x)[i];
  __syncthreads();
  const int M = q.M, lane = threadIdx.x % kClickPair, pairs = q.N * (q.N + 1) / 2;
  const int p = blockIdx.y * (blockDim.x / kClickPair) + threadIdx.x / kClickPair;
  int j, k;
  click_pair(min(p, pairs - 1), &j, &k);
  ClickEntry h{};
  if (q.U) {
    const cplx<double>* uj = q.U + (long long)q.S.m[j] * M;
    const cplx<double>* uk = q.U + (long long)q.S.m[k] * M;
    const int l_first = lane / kClickS * kClickL + lane % kClickS;
    ClickSum t;
    for (int l0 = 0; l0 < M; l0 += kClickG * kClickL) {
      constexpr int kT = kClickL / kClickS;
      cplx<double> x[kT], v[kT];
      double wa[kT], wb[kT];
#pragma unroll
      for (int i = 0; i < kT; ++i) {
        const int l = min(l0 + l_first + i * kClickS, M - 1);
        x[i] = uj[l];
        v[i] = uk[l];
        wa[i] = q.alpha[l];
        wb[i] = q.beta[l];
      }
      ClickSum run;
#pragma unroll
      for (int i = 0; i < kT; ++i)
        if (l0 + l_first + i * kClickS < M) run.step(x[i], v[i], wa[i], wb[i]);
      // the groups' runs in order (one beyond the last is zero)
#pragma unroll
      for (int g = 0; g < kClickG; ++g) t.add(run.from(g * kClickS + lane % kClickS));
    }
#pragma unroll
    for (int off = kClickS / 2; off > 0; off >>= 1) t.add(t.from(lane % kClickS + off));
    h = t.entry();
  } else {
    h = click_entry_dense(q, j, k);
  }
  if (lane == 0 && p < pairs) click_store(q, j, k, h, real_basis, roots);
}

// Many requests: a CTA per request and 128 pairs, a thread per pair, the rows of U staged
// in shared memory: nothing is summed across lanes (a warp per pair spends 20 of its FP64
// additions on that, more than on the products of a small state).  1500 requests of
// 5 .. 17 of 17 modes: 314 us with a warp per pair, 90 so.  From a request per SM on;
// fewer fill the chip better with lanes per pair.
__global__ void __launch_bounds__(128) batch_click_tile_kernel(const ClickReq* __restrict__ reqs, int real_basis,
                                                               void* __restrict__ roots) {
  __shared__ ClickReq q;
  __shared__ cplx<double> x[32][kClickL + 1];
  __shared__ double wa[kClickL], wb[kClickL];
  for (int i = threadIdx.x; i < (int)(sizeof(ClickReq) / 4); i += blockDim.x)
    reinterpret_cast<int*>(&q)[i] = reinterpret_cast<const int*>(reqs + blockIdx.x)[i];
  __syncthreads();
  const int p = blockIdx.y * blockDim.x + threadIdx.x, pairs = q.N * (q.N + 1) / 2, M = q.M;
  if ((int)(blockIdx.y * blockDim.x) >= pairs) return;
  int j, k;
  click_pair(min(p, pairs - 1), &j, &k);
  ClickEntry h{};
  if (q.U) {
    ClickSum t[kClickS];
    for (int l0 = 0; l0 < M; l0 += kClickL) {
      const int len = min(kClickL, M - l0);
      for (int e = threadIdx.x; e < q.N * kClickL; e += blockDim.x) {
        const int r = e / kClickL, c = e % kClickL;
        if (c < len) x[r][c] = q.U[(long long)q.S.m[r] * M + l0 + c];
      }
      if ((int)threadIdx.x < len) {
        wa[threadIdx.x] = q.alpha[l0 + threadIdx.x];
        wb[threadIdx.x] = q.beta[l0 + threadIdx.x];
      }
      __syncthreads();
      ClickSum run[kClickS];
      for (int c = 0; c < len; c += kClickS)
#pragma unroll
        for (int s = 0; s < kClickS; ++s)
          if (c + s < len) run[s].step(x[j][c + s], x[k][c + s], wa[c + s], wb[c + s]);
#pragma unroll
      for (int s = 0; s < kClickS; ++s) t[s].add(run[s]);
      __syncthreads();
    }
#pragma unroll
    for (int off = kClickS / 2; off > 0; off >>= 1)
#pragma unroll
      for (int s = 0; s < off; ++s) t[s].add(t[s + off]);
    h = t[0].entry();
  } else {
    h = click_entry_dense(q, j, k);
  }
  if (p < pairs) click_store(q, j, k, h, real_basis, roots);
}

// A-priori cancellation estimate of each tree: the ratio sum|t| / |Tor| the
// modes would have if they were independent, prod_j (g_j + 1) / |g_j - 1| with
// g_j = det(P_j)^(-1/2) of the mode's diagonal 2x2 block of the root (exact
// for independent modes; on Haar-random states it lies 0.3 to 17 orders of
// magnitude above the true ratio).  Output: log10 of it per tree (inf when a
// block has g = 1 or is not positive definite).
__global__ void kappa_estimate_kernel(const BatchTree* __restrict__ trees, int ntrees, const void* __restrict__ roots,
                                      int real_basis, double* __restrict__ log10_kappa) {
  // a warp per tree, a lane per mode: the logarithms (FP64, ~1 us each) side by side
  const int t = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const int lane = threadIdx.x & 31;
  if (t >= ntrees) return;
  const BatchTree tr = trees[t];
  double lk = 0.0;
  for (int j = lane; j < tr.n; j += 32) {
    const long long a = (long long)(2 * j) * (2 * j + 1) / 2 + 2 * j;        // tri(2j, 2j)
    const long long b = (long long)(2 * j + 1) * (2 * j + 2) / 2 + 2 * j;    // tri(2j+1, 2j)
    double det;
    if (real_basis) {
      const double* r = (const double*)roots + tr.root_off;
      det = r[a] * r[b + 1] - r[b] * r[b];
    } else {
      const cplx<double>* r = (const cplx<double>*)roots + tr.root_off;
      det = r[a].re * r[b + 1].re - (r[b].re * r[b].re + r[b].im * r[b].im);
    }
    const double g = det > 0.0 ? rsqrt(det) : 0.0;
    lk += det > 0.0 && g != 1.0 ? log10((g + 1.0) / fabs(g - 1.0)) : INFINITY;
  }
#pragma unroll
  for (int off = 16; off > 0; off >>= 1) lk += __shfl_down_sync(0xffffffffu, lk, off);
  if (lane == 0) log10_kappa[t] = lk;
}

// The engine of a precision and basis (fixed64: FP64 in 64-bit fixed point).
static gbs_status batch_variant(gbs_ctx* ctx, int prec, bool real, bool fixed64, int nt, const BatchTree* tr,
                                const void* roots, int* status, const TreeFinish& fin) {
  BatchEngine* e = nullptr;
  switch (prec) {
    case GBS_PREC_FP64: e = fixed64 ? batch_fxd_real : real ? batch_fp64_real : batch_fp64_cplx; break;
    case GBS_PREC_DD: e = real ? batch_dd_real : batch_dd_cplx; break;
    case GBS_PREC_TD: e = real ? batch_td_real : batch_td_cplx; break;
    case GBS_PREC_FP32_DIAG: e = real ? batch_fp32_real : batch_fp32_cplx; break;
    case GBS_PREC_FP64P:
      if (!real) return set_error(ctx, GBS_EINVAL, "the paired FP64 precision needs the real basis");
      e = batch_fp64p_real;
      break;
    case GBS_PREC_FXN:
    case GBS_PREC_FX:
    case GBS_PREC_FXW:
      if (!real) return set_error(ctx, GBS_EINVAL, "the fixed-point precision needs the real basis");
      e = prec == GBS_PREC_FXN ? batch_fxn_real : prec == GBS_PREC_FX ? batch_fx_real : batch_fxw_real;
      break;
    default: return set_error(ctx, GBS_EINVAL, "unknown precision");
  }
  return e(ctx, nt, tr, roots, status, batch_tune_for(ctx, fixed64 ? GBS_TUNE_FP64_FIXED : prec, real), fin);
}

gbs_status batch_eval(gbs_ctx* ctx, int prec, bool real, int ntrees, const BatchTree* trees, const void* roots_dev,
                      const double* logdet, ProbOut* host_out, int n_bounded) {
  if (ntrees <= 0) return GBS_OK;
  gbs_status st;
  const size_t n = (size_t)ntrees;
  auto r256 = [](size_t b) { return (b + 255) / 256 * 256; };
  const size_t bytes = r256(n * sizeof(ProbOut)) + r256(2 * n * sizeof(int));
  if ((st = dev_reserve(ctx, ctx->aux_dev, bytes))) return st;
  ProbOut* po = (ProbOut*)ctx->aux_dev.ptr;
  int* status = (int*)((unsigned char*)po + r256(n * sizeof(ProbOut)));  // then the counters
  if ((st = check_cuda(ctx, cudaMemsetAsync(status, 0, 2 * n * sizeof(int), ctx->stream), "memset"))) return st;
  const double u = unit_of(prec), extra = err_factor(prec, 1) - err_factor(GBS_PREC_TD, 1);
  std::vector<double> scale(n);
  for (size_t t = 0; t < n; ++t) scale[t] = std::exp(-0.5 * logdet[t]);
  // The bounded trees and the others, each on its engine, side by side and with one wait for
  // both: few trees are latency on either (16 FP64 requests of 8 .. 17 modes, half of them of
  // a state without a bound: 275 us in turn with a wait each, 264 with one, 186 side by side).
  struct Part {
    int first, count;
    bool fixed64;
    enum { kRun, kSplit, kFloat } todo;
  };
  const int nb = real && prec == GBS_PREC_FP64 ? n_bounded : 0;
  Part parts[2] = {{0, nb, true, Part::kRun}, {nb, ntrees - nb, false, Part::kRun}};
  gbs_status failed = GBS_OK;
  ctx->side_batch = nb > 0 && nb < ntrees;
  for (Part& p : parts) {
    if (p.count == 0 || failed) continue;
    ctx->batch_split = false;
    st = batch_variant(ctx, prec, real, p.fixed64, p.count, trees + p.first, roots_dev, status + p.first,
                       TreeFinish{scale.data() + p.first, u, extra, po + p.first, status + n + p.first,
                                  p.fixed64 && ctx->side_batch});
    if (st == GBS_ENOMEM && ctx->batch_split) {
      p.todo = Part::kSplit;
    } else if (st == GBS_ENOMEM && (p.fixed64 || ctx->side_batch)) {
      // by itself, on the floating engine: that keeps two levels where the fixed-point one
      // keeps all of a chunk, and the other part's workspace is free then
      p.todo = Part::kFloat;
    } else {
      failed = st;
    }
  }
  ctx->side_batch = false;
  if ((st = side_join(ctx))) return st;
  if (failed) return failed;
  if ((st = check_cuda(ctx, cudaMemcpyAsync(host_out, po, n * sizeof(ProbOut), cudaMemcpyDeviceToHost, ctx->stream),
                       "readback")) ||
      (st = stream_sync(ctx)))
    return st;
  for (KernelTimer* t : {&ctx->leaf_timer, &ctx->fx_leaf_timer}) {
    if (!t->pending) continue;
    float ms = 0.f;
    cudaEventElapsedTime(&ms, t->start, t->stop);
    ctx->leaf_timer.total_ms += ms;
    ctx->leaf_timer.count += 1;
    t->pending = false;
  }
  for (const Part& p : parts) {
    if (p.todo == Part::kRun) continue;
    // too large for one plan: the two halves in turn (a tree's result does not depend
    // on the rest of its batch, so the split changes no value)
    const int half = p.todo == Part::kSplit ? p.count / 2 : p.count;
    for (int i = 0, c = half; i < p.count; i += c, c = p.count - half) {
      const int k = p.first + i;
      if ((st = batch_eval(ctx, prec, real, c, trees + k, roots_dev, logdet + k, host_out + k,
                           p.fixed64 && p.todo == Part::kSplit ? c : 0)))
        return st;
    }
  }
  // a bounded tree whose values left the range after all: again in floating point
  std::vector<BatchTree> again;
  std::vector<double> ld;
  std::vector<int> which;
  for (int t = 0; t < nb; ++t)
    if (host_out[t].status == kStatusRange) {
      again.push_back(trees[t]);
      ld.push_back(logdet[t]);
      which.push_back(t);
    }
  if (!again.empty()) {
    std::vector<ProbOut> r(again.size());
    if ((st = batch_eval(ctx, prec, real, (int)again.size(), again.data(), roots_dev, ld.data(), r.data()))) return st;
    for (size_t i = 0; i < which.size(); ++i) host_out[which[i]] = r[i];
  }
  return GBS_OK;
}

// Click blocks of several (state, modes) requests into ctx->hbuf; fills trees[].
gbs_status batch_click_blocks(gbs_ctx* ctx, int nreq, const gbs_state* const* states, const int* const* modes,
                              const int* N, bool real, std::vector<BatchTree>& trees) {
  std::vector<ClickReq> reqs;
  trees.resize(nreq);
  long long ent = 0;
  int n_max = 0;
  for (int i = 0; i < nreq; ++i) {
    ClickReq q{};
    const gbs_state* st = states[i];
    q.U = st->has_factors ? (const cplx<double>*)st->U.ptr : nullptr;
    q.alpha = (const double*)st->alpha.ptr;
    q.beta = (const double*)st->beta.ptr;
    q.Sinv = (const cplx<double>*)st->Sinv.ptr;
    q.M = st->M;
    q.N = N[i];
    for (int j = 0; j < 32; ++j) q.S.m[j] = j < N[i] ? modes[i][j] : 0;
    q.root_off = ent;
    trees[i] = BatchTree{N[i], ent};
    n_max = std::max(n_max, N[i]);
    ent += (long long)N[i] * (2 * N[i] + 1);  // sym(2N)
    if (N[i] > 0) reqs.push_back(q);
  }
  gbs_status st;
  if ((st = dev_reserve(ctx, ctx->hbuf, (size_t)std::max(1LL, ent) * (real ? 8 : 16)))) return st;
  if (reqs.empty()) return GBS_OK;
  const void* d = nullptr;
  if ((st = stage(ctx, reqs.data(), reqs.size() * sizeof(ClickReq), &d))) return st;
  const int pairs = n_max * (n_max + 1) / 2;
  const bool many = (int)reqs.size() >= ctx->sm_count;
  const int per_cta = many ? 128 : 128 / kClickPair;
  (many ? batch_click_tile_kernel : batch_click_block_kernel)<<<
      dim3((unsigned)reqs.size(), (unsigned)((pairs + per_cta - 1) / per_cta)), 128, 0, ctx->stream>>>(
      (const ClickReq*)d, real ? 1 : 0, ctx->hbuf.ptr);
  count_launch(ctx);
  return check_cuda(ctx, cudaGetLastError(), "click blocks");
}

static void fill(gbs_prob* out, const ProbOut& r, int prec, bool real, double logdet) {
  out->p_hi = r.p_hi;
  out->p_lo = r.p_lo;
  for (int i = 0; i < 3; ++i) out->tor[i] = r.tor[i];
  out->abs_sum = r.abs_sum;
  out->kappa = r.kappa;
  out->err_bound = r.err;
  out->logdet_sigma = logdet;
  out->prec_used = prec;
  out->basis_used = real ? GBS_BASIS_REAL : GBS_BASIS_COMPLEX;
  out->status = r.status == kStatusNotPD ? GBS_ENOTPD : r.status == kStatusRange ? GBS_EPRECISION : GBS_OK;
}

// Probabilities of a batch of requests with the precision ladder; out[] per request.
gbs_status probs_batch(gbs_ctx* ctx, int nreq, const gbs_state* const* states, const int* const* modes, const int* N,
                       int prec, int basis, double rel_tol, gbs_prob* out) {
  const bool real = basis != GBS_BASIS_COMPLEX;
  gbs_status st;
  if ((st = stage_begin(ctx, (size_t)nreq * 8192 + (1 << 16)))) return st;
  std::vector<BatchTree> trees;
  if ((st = batch_click_blocks(ctx, nreq, states, modes, N, real, trees))) return st;
  const double tol = rel_tol > 0 ? rel_tol : 1e-10;
  // requests still to evaluate (N == 0 needs no tree: Tor = 1)
  std::vector<int> todo;
  for (int i = 0; i < nreq; ++i) {
    if (N[i] == 0) {
      memset(&out[i], 0, sizeof(gbs_prob));
      out[i].p_hi = exp(-0.5 * states[i]->logdet_sigma);
      out[i].tor[0] = 1.0;
      out[i].abs_sum = 1.0;
      out[i].kappa = 1.0;
      out[i].logdet_sigma = states[i]->logdet_sigma;
      out[i].prec_used = prec == GBS_PREC_AUTO ? GBS_PREC_FP64 : prec;
      out[i].basis_used = real ? GBS_BASIS_REAL : GBS_BASIS_COMPLEX;
    } else {
      todo.push_back(i);
    }
  }
  // AUTO: FP64; then FP64 with the last two levels cancellation-free (real
  // basis) for the requests whose FP64 estimate missed rel_tol by at most
  // kPairReach (the grouping's estimate is 1e1 to 1e3 below FP64's on the
  // states it was measured on); then fixed point (160, then 192 fraction bits) where the
  // state bounds the tree (real basis), then triple-double.  A request moves
  // on while its error estimate misses rel_tol or its fixed-point tree left the
  // range.  The narrow fixed point (128 fraction bits) comes before FX for the
  // requests whose earlier rungs bound |p| away from zero well enough to
  // predict its estimate (FP64's scaled by 2^-55) within rel_tol with a factor
  // 2 of margin; without such a bound a miss would cost ~0.7 of FX on top.
  // Trees of kSkip64 or more modes skip FP64 unless the a-priori cancellation
  // estimate (kappa_estimate_kernel) leaves it within kPairReach of rel_tol:
  // there FP64 almost never certifies and costs ~0.2 of FX for nothing.  The
  // estimate is exact for independent modes but runs up to 17 orders of
  // magnitude high on correlated ones, so smaller trees keep the FP64 rung
  // (cheap, and the bound on |p| it gives admits them to the narrow fixed
  // point); a tree that skipped FP64 goes to the narrow fixed point only when
  // the estimate itself predicts success.  Only trees of kSkip64 or more modes
  // consult the estimate, so it is computed only when the batch holds one, and
  // a request's rungs never depend on what it is batched with.
  constexpr double kPairReach = 1e3;
  constexpr int kSkip64 = 16;
  const int ladder[6] = {GBS_PREC_FP64, GBS_PREC_FP64P, GBS_PREC_FXN, GBS_PREC_FX, GBS_PREC_FXW, GBS_PREC_TD};
  const int steps = prec == GBS_PREC_AUTO ? 6 : 1;
  bool uncertified = false;
  std::vector<double> err64(nreq, INFINITY), p_low(nreq, 0.0);  // FP64 estimate, lower bound on |p|
  std::vector<double> lk(nreq, INFINITY);  // log10 of the a-priori cancellation estimate
  bool need_estimate = false;  // only trees of kSkip64+ modes use it (to skip FP64, and then for FXN)
  for (int i : todo) need_estimate |= N[i] >= kSkip64;
  if (prec == GBS_PREC_AUTO && need_estimate) {
    std::vector<BatchTree> tt(todo.size());
    for (size_t i = 0; i < todo.size(); ++i) tt[i] = trees[todo[i]];
    std::vector<double> est(todo.size(), 0.0);
    const void *d_tt = nullptr, *d_est = nullptr;
    if ((st = stage(ctx, tt.data(), tt.size() * sizeof(BatchTree), &d_tt)) ||
        (st = stage(ctx, est.data(), est.size() * sizeof(double), &d_est)))
      return st;
    kappa_estimate_kernel<<<(unsigned)((todo.size() + 3) / 4), 128, 0, ctx->stream>>>(
        (const BatchTree*)d_tt, (int)todo.size(), ctx->hbuf.ptr, real ? 1 : 0, (double*)d_est);
    count_launch(ctx);
    if ((st = check_cuda(ctx, cudaMemcpyAsync(est.data(), d_est, est.size() * sizeof(double), cudaMemcpyDeviceToHost,
                                              ctx->stream),
                         "kappa estimate")) ||
        (st = stream_sync(ctx)))
      return st;
    for (size_t i = 0; i < todo.size(); ++i) lk[todo[i]] = est[i];
  }
  std::vector<char> ran64(nreq, 0);
  for (int k = 0; k < steps && !todo.empty(); ++k) {
    const int pr = prec == GBS_PREC_AUTO ? ladder[k] : prec;
    std::vector<int> run, next;
    for (int i : todo) {
      const double l4n = std::log10(4.0 * std::max(N[i], 1));
      if (prec == GBS_PREC_AUTO && pr == GBS_PREC_FP64 && N[i] >= kSkip64 &&
          !(l4n - 53.0 * std::log10(2.0) + lk[i] <= std::log10(kPairReach * tol))) {
        next.push_back(i);
        continue;
      }
      if (prec == GBS_PREC_AUTO && pr == GBS_PREC_FP64P &&
          !(real && ran64[i] && out[i].err_bound <= kPairReach * tol * fabs(out[i].p_hi))) {
        next.push_back(i);
        continue;
      }
      if (prec == GBS_PREC_AUTO && pr == GBS_PREC_FXN && !(2.0 * err64[i] * 0x1p-55 <= tol * p_low[i]) &&
          !(N[i] >= kSkip64 && std::log10(2.0) + l4n - 108.0 * std::log10(2.0) + lk[i] <= std::log10(tol))) {
        next.push_back(i);
        continue;
      }
      if (is_fixed_point(pr) && !(real && fx_ok_inverse(states[i], N[i]))) {
        if (prec == GBS_PREC_AUTO) {
          next.push_back(i);
          continue;
        }
        return set_error(ctx, GBS_EPRECISION, "the state does not bound the fixed-point tree (or basis not real)");
      }
      run.push_back(i);
    }
    // FP64: the trees their states bound first, in 64-bit fixed point
    std::stable_partition(run.begin(), run.end(), [&](int i) {
      return pr == GBS_PREC_FP64 && real && fxd_ok_inverse(states[i], N[i]);
    });
    size_t nb = 0;
    while (nb < run.size() && pr == GBS_PREC_FP64 && real && fxd_ok_inverse(states[run[nb]], N[run[nb]])) ++nb;
    std::vector<BatchTree> sub(run.size());
    std::vector<double> ld(run.size());
    for (size_t i = 0; i < run.size(); ++i) {
      sub[i] = trees[run[i]];
      ld[i] = states[run[i]]->logdet_sigma;
    }
    std::vector<ProbOut> res(run.size());
    if ((st = batch_eval(ctx, pr, real, (int)run.size(), sub.data(), ctx->hbuf.ptr, ld.data(), res.data(), (int)nb)))
      return st;
    for (size_t i = 0; i < run.size(); ++i) {
      fill(&out[run[i]], res[i], pr, real, ld[i]);
      if (prec != GBS_PREC_AUTO) continue;
      if (pr == GBS_PREC_FP64) {
        err64[run[i]] = res[i].err;
        ran64[run[i]] = 1;
      }
      if (res[i].status == 0) p_low[run[i]] = std::max(p_low[run[i]], fabs(res[i].p_hi) - res[i].err);
      const bool missed = res[i].status == 0 && !(res[i].err <= tol * fabs(res[i].p_hi));
      // triple-double (u = 2^-152) cannot improve on a wide fixed-point result
      // (2^-158): such a request stops here, uncertified
      if (missed && pr == GBS_PREC_FXW)
        uncertified = true;
      else if (res[i].status == kStatusRange || missed)
        next.push_back(run[i]);
    }
    std::sort(next.begin(), next.end());
    todo.swap(next);
    if (k == steps - 1 && !todo.empty()) uncertified = true;
  }
  for (int i = 0; i < nreq; ++i) {
    if (out[i].status == GBS_ENOTPD) return set_error(ctx, GBS_ENOTPD, "a pivot block is not positive definite");
    if (out[i].status) return set_error(ctx, out[i].status, "a fixed-point tree left its range");
  }
  if (uncertified) return set_error(ctx, GBS_EPRECISION, "the triple-double error estimate exceeds rel_tol");
  return GBS_OK;
}

}  // namespace gbs

using namespace gbs;

// Times the candidate shapes of tune[shape][real] on the trees (all on leading blocks of one
// host root) and keeps the fastest.
static gbs_status autotune_shape(gbs_ctx* ctx, int shape, bool real, const std::vector<double>& root,
                                 const std::vector<BatchTree>& trees, std::string* rep) {
  const bool fixed64 = shape == GBS_TUNE_FP64_FIXED, fixed = fixed64 || is_fixed_point(shape);
  const int prec = fixed64 ? (int)GBS_PREC_FP64 : shape, n_trees = (int)trees.size();
  const std::vector<double> zeros(n_trees, 0.0);
  std::vector<ProbOut> outs(n_trees);
  BatchTune& slot = ctx->tune[shape][real ? 1 : 0];
  const BatchTune saved = slot;
  BatchTune best = saved;
  double best_ms = 1e30;
  gbs_status st;
  cudaEvent_t e0, e1;
  cudaEventCreate(&e0);
  cudaEventCreate(&e1);
  const int subs[] = {0, 2, 3, 4, 5, 6, 7};
  const int tops[] = {6, 8, 9, 10};
  const int grids[] = {0, 8};
  const long long lts[] = {1LL << 17, 1LL << 19};
  const int mids[] = {0, 4, 5};
  for (int me : mids)
  for (int qd = 0; qd < 2; ++qd)
  for (int se : subs)
    for (int dt : tops)
      for (int gr : grids)
        for (long long lt : lts) {
          BatchTune cand;
          cand.sub_e = se;
          cand.d_top = dt;
          cand.leaf_grid_per_sm = gr;
          cand.level_threads = lt;
          cand.q_drop = qd;
          cand.mid_e = me;
          // only d_top and q_drop act on the fixed-point engine: one candidate for the rest
          if (fixed && (me != mids[0] || se != subs[0] || gr != grids[0] || lt != lts[0])) continue;
          slot = cand;
          float ms_best = 1e30f;
          for (int rep_i = 0; rep_i < 3; ++rep_i) {
            if ((st = stage_begin(ctx, root.size() * 8 + (1 << 16)))) goto done;
            const void* d = nullptr;
            if ((st = stage(ctx, root.data(), root.size() * 8, &d))) goto done;
            cudaEventRecord(e0, ctx->stream);
            if ((st = batch_eval(ctx, prec, real, n_trees, trees.data(), d, zeros.data(), outs.data(),
                                 fixed64 ? n_trees : 0)))
              goto done;
            cudaEventRecord(e1, ctx->stream);
            cudaEventSynchronize(e1);
            float ms = 0.f;
            cudaEventElapsedTime(&ms, e0, e1);
            if (rep_i > 0 && ms < ms_best) ms_best = ms;  // the first run warms up
          }
          char buf[192];
          snprintf(buf, sizeof buf,
                   "%s{\"sub_e\":%d,\"d_top\":%d,\"grid_per_sm\":%d,\"level_threads\":%lld,\"q_drop\":%d,"
                   "\"mid_e\":%d,\"ms\":%.4f}",
                   rep->empty() ? "" : ",", se, dt, gr, lt, qd, me, ms_best);
          *rep += buf;
          if (ms_best < best_ms) {
            best_ms = ms_best;
            best = cand;
          }
        }
  st = GBS_OK;
done:
  cudaEventDestroy(e0);
  cudaEventDestroy(e1);
  slot = st == GBS_OK ? best : saved;
  return st;
}

// Whether (prec, basis) names a launch shape.
static bool valid_shape(int prec, int basis) {
  return prec >= GBS_PREC_FP64 && prec <= kTuneLast && !(prec == GBS_TUNE_FP64_FIXED && basis == GBS_BASIS_COMPLEX);
}

extern "C" gbs_status gbs_autotune(gbs_ctx* ctx, int prec, int basis, int n, int n_trees, char* report,
                                   size_t report_len) {
  if (!ctx || !valid_shape(prec, basis) || n < 6 || n > 28 || n_trees < 1 || n_trees > 64) return GBS_EINVAL;
  if (prec >= GBS_PREC_FX && basis == GBS_BASIS_COMPLEX) return GBS_EINVAL;
  std::lock_guard<std::mutex> g(ctx->mu);
  cudaSetDevice(ctx->device);
  const bool real = basis != GBS_BASIS_COMPLEX;
  // A synthetic well-conditioned positive-definite root (the timing does not
  // depend on the values): identity plus a small symmetric perturbation.
  const int D = 2 * n, ne = D * (D + 1) / 2;
  std::vector<double> root(ne * (real ? 1 : 2), 0.0);
  unsigned long long x = 0x9E3779B97F4A7C15ull;
  for (int a = 0; a < D; ++a)
    for (int b = 0; b <= a; ++b) {
      const int t = a * (a + 1) / 2 + b;
      x ^= x << 13; x ^= x >> 7; x ^= x << 17;
      const double v = (a == b) ? 1.0 : 0.02 * ((double)(x >> 11) * 0x1p-53 - 0.5);
      if (real) root[t] = v; else { root[2 * t] = v; root[2 * t + 1] = (a == b) ? 0.0 : 0.5 * v; }
    }
  // n_trees trees of n, n-1, ... modes (at least 6), all on leading blocks of the one root
  std::vector<BatchTree> trees(n_trees);
  for (int i = 0; i < n_trees; ++i) trees[i] = BatchTree{std::max(6, n - i), 0};
  std::string rep, rep64;
  gbs_status st = autotune_shape(ctx, prec, real, root, trees, &rep);
  // FP64 calls run on either engine
  if (st == GBS_OK && prec == GBS_PREC_FP64 && real)
    st = autotune_shape(ctx, GBS_TUNE_FP64_FIXED, real, root, trees, &rep64);
  if (report && report_len) snprintf(report, report_len, "[%s]", rep.c_str());
  return st;
}

extern "C" gbs_status gbs_get_tuning(gbs_ctx* ctx, int prec, int basis, int* sub_e, int* d_top, int* grid_per_sm,
                                     long long* level_threads, int* q_drop, int* mid_e) {
  if (!ctx || !valid_shape(prec, basis)) return GBS_EINVAL;
  const BatchTune& t = ctx->tune[prec][basis != GBS_BASIS_COMPLEX ? 1 : 0];
  if (sub_e) *sub_e = t.sub_e;
  if (d_top) *d_top = t.d_top;
  if (grid_per_sm) *grid_per_sm = t.leaf_grid_per_sm;
  if (level_threads) *level_threads = t.level_threads;
  if (q_drop) *q_drop = t.q_drop;
  if (mid_e) *mid_e = t.mid_e;
  return GBS_OK;
}

extern "C" gbs_status gbs_set_tuning(gbs_ctx* ctx, int prec, int basis, int sub_e, int d_top, int grid_per_sm,
                                     long long level_threads, int q_drop, int mid_e) {
  if (!ctx || !valid_shape(prec, basis) || sub_e < 0 || sub_e > 7 || d_top < 0 || d_top > 16 || grid_per_sm < 0 ||
      level_threads < 1 || q_drop < 0 || q_drop > 2 || mid_e < 0 || mid_e > 8)
    return GBS_EINVAL;
  std::lock_guard<std::mutex> g(ctx->mu);
  BatchTune& t = ctx->tune[prec][basis != GBS_BASIS_COMPLEX ? 1 : 0];
  t.sub_e = sub_e;
  t.d_top = d_top;
  t.leaf_grid_per_sm = grid_per_sm;
  t.level_threads = level_threads;
  t.q_drop = q_drop;
  t.mid_e = mid_e;
  return GBS_OK;
}

extern "C" gbs_status gbs_torontonian_batch(gbs_ctx* ctx, int n_req, const gbs_state* const* states,
                                            const int* modes, const int* N_per, int prec, int basis, double rel_tol,
                                            gbs_prob* out) {
  if (!ctx || n_req < 0 || (n_req > 0 && (!states || !N_per || !out))) return GBS_EINVAL;
  if (prec < GBS_PREC_AUTO || prec > kPrecLast) return GBS_EINVAL;
  std::lock_guard<std::mutex> g(ctx->mu);
  cudaSetDevice(ctx->device);
  std::vector<const int*> mp(n_req);
  long long off = 0;
  for (int i = 0; i < n_req; ++i) {
    if (!states[i] || states[i]->ctx != ctx) return set_error(ctx, GBS_EINVAL, "state of another context");
    mp[i] = modes ? modes + off : nullptr;
    if (const gbs_status st = validate_modes(ctx, mp[i], N_per[i], states[i]->M)) return st;
    off += N_per[i];
  }
  if (n_req == 0) return GBS_OK;
  return probs_batch(ctx, n_req, states, mp.data(), N_per, prec, basis, rel_tol, out);
}
