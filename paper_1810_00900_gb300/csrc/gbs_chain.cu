// Whole steps of the chain-rule sampler in one CTA per trajectory.
//
// While a trajectory has few clicks a step is latency only: a gather, a small tree, a
// read-back, a decision, a read-back and two conditioning launches made ~110 us, of
// which the tree was 15-35.  Here a CTA takes a trajectory through up to kChainSteps
// steps: it picks the precision as sampler_advance does, forms the tree in shared memory
// (fx_cta_tree, in the type of that precision), checks the error bound, decides, and
// conditions Sigma' -- the same functions and order as the launches, so the bits are the
// same.  It stops, without having changed anything of that step, when the step is not
// for it: too many modes, another precision, a bound that misses the tolerance or a
// value out of range; the next call then takes that step the other way.
//
// What bounds it is latency: at M = 100 a step takes ~20 us, about 10 in the tree's
// phases, 4 in the decision's chains of FP64 operations, the rest in the conditioning
// (~A^2/2 FP64 updates of two FMAs each, at 2 per clock and SM: 8 us on one SM, so the
// CTAs of a cluster share it).  8 postselected samples of a 100-mode graph state: 131 ms
// with a launch per operation, 39 here; 64 free samples of 30 modes: 5.4 and 3.2.  At M =
// 200 the conditioning on one SM is up to 40 us a step; with a cluster 24 trajectories of
// 200 modes take 39.4 ms, 42.8 without.
#include <cooperative_groups.h>

#include <algorithm>
#include <chrono>
#include <cstring>
#include <vector>

#include "gbs_fxtree.cuh"
#include "gbs_internal.h"
#include "gbs_sampler_dev.cuh"

namespace gbs {

namespace {

// Up to kChainAnyM modes with any number of trajectories, up to kChainMaxM with at most one
// per two SMs: beyond, the chip's SMs are not all busy conditioning where the launches spread
// every trajectory over all of them.  10 forced clicks, ms with launches / here: 448 modes, 1, 8, 64,
// 160 trajectories 45 / 17, 54 / 22, 84 / 44, 119 / 105; 800 modes 90 / 47, 110 / 54, 222 / 166,
// 372 / 481; 1000 modes, 64: 349 / 291.
constexpr int kChainAnyM = 448, kChainMaxM = 1024;

// Modes a CTA's tree may have in the type of a precision.
GBS_HD_INLINE int chain_modes(int prec) { return prec == GBS_PREC_FP64 || prec == GBS_PREC_FXN ? 10 : 9; }
GBS_HD_INLINE bool chain_prec(int prec) {
  return prec == GBS_PREC_FP64 || prec == GBS_PREC_FXN || prec == GBS_PREC_FX || prec == GBS_PREC_FXW;
}

struct ChainJob {
  double* sig;
  int* clicks;
  double* dcarry;
  unsigned long long seed;
  double kappa_prev, relD;
  int M, sample, attempt, N_post, step, m, need_full, prec, is_forced, pad;
  uint32_t forced[(kChainMaxM + 31) / 32];  // bit k: mode k is forced to click
};

enum { kChainMore = 0, kChainDone = 1, kChainRejected = 2, kChainHost = 3 };

struct ChainOut {
  double kappa_prev, relD;
  int steps, m, need_full, code, near_ties, uncertified;
  int trees[6];
  unsigned clicked;  // bit i: the i-th of these steps was a click
  int pad;
  double p0[kChainSteps];
};

// The trajectory's state between steps and what thread 0 tells the others.
struct ChainShared {
  int step, m, need_full, prec, stop, click, bad, go, k;
  double kappa_prev, relD, dcarry[3];
  int clicks[40];
  ModePivot pv;
  td tor;
  double abs_sum, dp, kappa_next, relD_next;
};

template <class E>
__device__ __noinline__ void chain_tree(unsigned char* smem, const double* sig, long long D, const int* clicks, int m, int k,
                                        bool half, int n, const ModePivot& pivot, TreeOut* out, int* bad) {
  const ModePivot pv = pivot;
  bool ok = true;
  const auto sum =
      fx_cta_tree<E, true>(smem, n, 0, 0u, [&](int i) { return step_root(sig, D, clicks, m, k, half, pv, i); }, ok);
  if (!ok) *bad = 1;
  if (threadIdx.x == 0) {
    fx_store3(sum.inc, out->inc);
    fx_store3(sum.exc, out->exc);
    out->abs = to_double(sum.abs);
  }
  __syncthreads();
}

// Conditions the active rows on mode k dark (its clicked modes are those before it): this
// CTA's share of the rows, one of `parts`.  No row or column of mode k changes, so every CTA
// forms the factors from Sigma' itself.
__device__ __forceinline__ void chain_condition(unsigned char* smem, double* sig, long long D, const ChainShared& st,
                                                int k, int m, int part, int parts) {
  const int tid = threadIdx.x, lane = tid & 31;
  const int A = 2 * k + 2 * m;
  const long long rk = 2LL * k;
  double* u0 = reinterpret_cast<double*>(smem);
  double *u1 = u0 + A, *l0 = u1 + A, *l1 = l0 + A;
  int* row = reinterpret_cast<int*>(l1 + A);
  const ModePivot pv = st.pv;
  for (int i = tid; i < A; i += blockDim.x) {
    const int ri = i < 2 * k ? i : 2 * st.clicks[(i - 2 * k) >> 1] + ((i - 2 * k) & 1);
    const double a0 = sig_at(sig, D, ri, rk), a1 = sig_at(sig, D, ri, rk + 1);
    row[i] = ri;
    u0[i] = a0;
    u1[i] = a1;
    l0[i] = fma(a0, pv.q00, a1 * pv.q10);
    l1[i] = fma(a0, pv.q10, a1 * pv.q11);
  }
  __syncthreads();
  // a warp per row; four of its entries are in flight at a time (one at a time, the
  // loads' latency was most of a step)
  for (int i = (tid >> 5) * parts + part; i < A; i += (blockDim.x >> 5) * parts) {
    const int ri = row[i];
    const double x0 = l0[i], x1 = l1[i];
    double* dst = sig + (long long)ri * D;
    const int jmax = i < 2 * k ? i + 1 : A;
    for (int c0 = lane; c0 < jmax; c0 += 128) {
      double x[4];
      int rc[4];
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        const int c = c0 + 32 * q;
        rc[q] = c < jmax ? row[c] : ri + 1;
        if (rc[q] <= ri) x[q] = dst[rc[q]];
      }
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        const int c = c0 + 32 * q;
        if (rc[q] <= ri) dst[rc[q]] = fma(-x0, u0[c], fma(-x1, u1[c], x[q]));
      }
    }
  }
}

// A cluster per trajectory: its first CTA takes the steps, the others (chain_cluster) only
// their share of the conditioning.  All of a cluster's CTAs pass the same barriers: two per
// conditioning, two at the end.
__global__ void __launch_bounds__(512) chain_kernel(const ChainJob* __restrict__ jobs, ChainOut* __restrict__ outs) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ ChainShared st;
  __shared__ TreeOut tree;
  const cooperative_groups::cluster_group cluster = cooperative_groups::this_cluster();
  const int job = (int)(blockIdx.x / cluster.num_blocks());
  const ChainJob j = jobs[job];
  ChainOut* out = outs + job;
  const long long D = 2LL * j.M;
  const int tid = threadIdx.x;
  if (cluster.block_rank() != 0) {
    const int* lead = reinterpret_cast<const int*>(cluster.map_shared_rank(&st, 0));
    for (;;) {
      cluster.sync();
      for (int i = tid; i < (int)(sizeof(ChainShared) / 4); i += blockDim.x) reinterpret_cast<int*>(&st)[i] = lead[i];
      __syncthreads();
      if (!st.go) break;
      chain_condition(smem_raw, j.sig, D, st, st.k, st.m, (int)cluster.block_rank(), (int)cluster.num_blocks());
      cluster.sync();
    }
    cluster.sync();
    return;
  }
  int trees[6] = {0, 0, 0, 0, 0, 0}, near_ties = 0, uncertified = 0, steps = 0, code = kChainMore;  // thread 0's
  unsigned clicked = 0u;
  if (tid < j.m) st.clicks[tid] = j.clicks[tid];
  if (tid == 0) {
    st.step = j.step;
    st.m = j.m;
    st.need_full = j.need_full;
    st.kappa_prev = j.kappa_prev;
    st.relD = j.relD;
    for (int i = 0; i < 3; ++i) st.dcarry[i] = j.dcarry[i];
  }
  for (int it = 0; it < kChainSteps; ++it) {
    __syncthreads();
    const int step = st.step, m = st.m, k = j.M - 1 - step;
    const bool half = !st.need_full;
    const int n = half ? m : m + 1;
    if (tid == 0) {
      st.prec = j.prec != GBS_PREC_AUTO ? j.prec : sampler_pick(true, st.kappa_prev * (half ? 1.5 : 8.0), n);
      st.bad = 0;
    }
    if (tid == 64) st.pv = mode_pivot(j.sig, D, k);
    __syncthreads();
    const int prec = st.prec;
    if (!chain_prec(prec) || n > chain_modes(prec)) {
      code = kChainHost;
      break;
    }
    if (n > 0) {
      switch (prec) {
        case GBS_PREC_FP64: chain_tree<fxd>(smem_raw, j.sig, D, st.clicks, m, k, half, n, st.pv, &tree, &st.bad); break;
        case GBS_PREC_FXN: chain_tree<fxn4>(smem_raw, j.sig, D, st.clicks, m, k, half, n, st.pv, &tree, &st.bad); break;
        case GBS_PREC_FX: chain_tree<fx>(smem_raw, j.sig, D, st.clicks, m, k, half, n, st.pv, &tree, &st.bad); break;
        default: chain_tree<fxw>(smem_raw, j.sig, D, st.clicks, m, k, half, n, st.pv, &tree, &st.bad); break;
      }
    }
    if (tid == 0) {
      st.tor = n > 0 ? td{tree.inc[0], tree.inc[1], tree.inc[2]} + td{tree.exc[0], tree.exc[1], tree.exc[2]}
                     : td{1.0, 0.0, 0.0};  // no clicks yet: Tor = 1 exactly
      st.abs_sum = n > 0 ? tree.abs : 1.0;
    }
    __syncthreads();
    // The scalar work is chains of FP64 operations: the checks of sampler_advance on one
    // warp's thread, the decision on another's.
    if (tid == 32) {
      const double u = unit_of(prec), f = err_factor(prec, n);
      const double at = fabs(st.tor.x0), exc = n > 0 ? fabs(tree.exc[0]) : 0.0, inc = n > 0 ? fabs(tree.inc[0]) : 0.0;
      if (half) {
        st.kappa_next = st.abs_sum / fmax(at, 1e-300);
        st.relD_next = f * u * st.kappa_next + 2e-16;  // the carried D is (-1)^m Tor_k
        st.dp = (n > 0 ? f * u * st.abs_sum / fmax(at, 1e-300) : 0.0) + 2e-16 + st.relD;
      } else {
        st.kappa_next = st.abs_sum / fmax(fmin(exc, inc), 1e-300);
        st.relD_next = f * u * st.abs_sum / fmax(inc, 1e-300) + 4e-16;
        st.dp = f * u * st.abs_sum * (1.0 + (exc > 0 ? inc / exc : INFINITY)) / fmax(exc, 1e-300);
      }
    }
    Decision d{};
    double carry[3];
    if (tid == 0) {
      const double t3[3] = {st.tor.x0, st.tor.x1, st.tor.x2};
      const int forced = j.is_forced ? (int)((j.forced[k >> 5] >> (k & 31)) & 1u) : -1;
      for (int i = 0; i < 3; ++i) carry[i] = st.dcarry[i];
      d = decide_step(half ? t3 : tree.inc, tree.exc, carry, half, m, st.pv, forced, j.seed, step, j.sample, j.attempt);
    }
    __syncthreads();
    if (tid == 0) {
      const bool sure = st.dp < kSampleTol;
      st.stop = st.bad || (!sure && j.prec == GBS_PREC_AUTO);
      if (!st.stop) {
        if (n > 0) trees[stat_slot(prec)]++;
        if (!sure) uncertified++;
        st.kappa_prev = st.kappa_next;
        st.relD = st.relD_next;
        out->p0[it] = d.p0;
        near_ties += d.near_tie;
        st.click = d.click;
        st.need_full = d.click;
        if (d.click) {
          clicked |= 1u << it;
          st.clicks[m] = k;
          j.clicks[m] = k;
          st.m = m + 1;
        } else {
          for (int i = 0; i < 3; ++i) j.dcarry[i] = st.dcarry[i] = carry[i];
        }
        steps = it + 1;
        const int m2 = st.m;
        if (!j.is_forced && ((j.N_post > 0 && (m2 > j.N_post || m2 + k < j.N_post)) || m2 > 31)) {
          code = kChainRejected;
          st.stop = 1;
        } else {
          st.step = step + 1;
          if (k == 0) {
            code = kChainDone;
            st.stop = 1;
          }
        }
      } else {
        code = kChainHost;
      }
    }
    __syncthreads();
    if (st.stop) break;
    if (!st.click) {
      if (cluster.num_blocks() > 1) {
        if (tid == 0) {
          st.go = 1;
          st.k = k;
        }
        cluster.sync();
      }
      chain_condition(smem_raw, j.sig, D, st, k, m, 0, (int)cluster.num_blocks());
      if (cluster.num_blocks() > 1) cluster.sync();
    }
  }
  if (cluster.num_blocks() > 1) {
    if (tid == 0) st.go = 0;
    cluster.sync();
  }
  if (tid == 0) {
    out->kappa_prev = st.kappa_prev;
    out->relD = st.relD;
    out->steps = steps;
    out->m = st.m;
    out->need_full = st.need_full;
    out->code = code;
    out->near_ties = near_ties;
    out->uncertified = uncertified;
    for (int i = 0; i < 6; ++i) out->trees[i] = trees[i];
    out->clicked = clicked;
  }
  if (cluster.num_blocks() > 1) cluster.sync();  // the others have read st.go
}

}  // namespace

bool chain_eligible(const gbs_ctx* ctx, const Trajectory& t, int prec, size_t n_traj) {
  if (t.M > (2 * n_traj <= (size_t)ctx->sm_count ? kChainMaxM : kChainAnyM) || !fx_ok_sigma(t.st, 32)) return false;
  const bool half = !t.need_full;
  const int n = half ? t.m : t.m + 1;
  const int p = prec != GBS_PREC_AUTO ? prec : sampler_pick(true, t.kappa_prev * (half ? 1.5 : 8.0), n);
  return chain_prec(p) && n <= chain_modes(p);
}

gbs_status chain_advance(gbs_ctx* ctx, const std::vector<Trajectory*>& jobs, int prec, gbs_sample_stats& stt) {
  const size_t T = jobs.size();
  gbs_status e;
  if ((e = stage_begin(ctx, T * sizeof(ChainJob)))) return e;
  std::vector<ChainJob> in(T);
  int m_max = 0, M_max = 0;
  for (size_t i = 0; i < T; ++i) {
    const Trajectory* t = jobs[i];
    ChainJob& j = in[i];
    memset(&j, 0, sizeof j);
    j.sig = t->sig;
    j.clicks = t->clicks;
    j.dcarry = t->dcarry;
    j.seed = t->seed;
    j.kappa_prev = t->kappa_prev;
    j.relD = t->relD;
    j.M = t->M;
    j.sample = t->sample;
    j.attempt = t->attempt;
    j.N_post = t->N_post;
    j.step = t->step;
    j.m = t->m;
    j.need_full = t->need_full;
    j.prec = prec;
    j.is_forced = t->forced.empty() ? 0 : 1;
    for (int k = 0; k < (int)t->forced.size(); ++k)
      if (t->forced[k]) j.forced[k >> 5] |= 1u << (k & 31);
    m_max = std::max(m_max, t->m);
    M_max = std::max(M_max, t->M);
  }
  const void* d_in = nullptr;
  if ((e = stage(ctx, in.data(), T * sizeof(ChainJob), &d_in))) return e;
  if ((e = dev_reserve(ctx, ctx->out, T * sizeof(ChainOut)))) return e;
  ChainOut* d_out = (ChainOut*)ctx->out.ptr;
  // the largest tree any of the types may meet, and the conditioning's rows
  const int tree_words = std::max(std::max(fx_small_words(10, 10, 3, 5), fx_small_words(10, 10, 5, 6)),
                                  std::max(fx_small_words(9, 9, 6, 7), fx_small_words(9, 9, 7, 8)));
  const size_t smem = std::max((size_t)tree_words * 4, (size_t)(2 * M_max + 2) * (4 * sizeof(double) + sizeof(int)));
  if ((e = allow_smem(ctx, chain_kernel, smem, "chain smem"))) return e;
  const auto t0 = std::chrono::steady_clock::now();
  // CTAs per trajectory: as many as are resident at once, up to a portable cluster's 8 (18
  // trajectories of 230 modes: 14.8 ms with clusters of 8, which do not all fit, 11.6 with 4).
  // 8 trajectories of a 100-mode graph state, ms: 44.7 with one, 43.7, 41.5, 40.5 with 2, 4,
  // 8; 24 of 200 modes 42.8, 41.4, 40.1; 64 of 30 modes 3.3 with one and two.
  cudaLaunchAttribute attr;
  attr.id = cudaLaunchAttributeClusterDimension;
  attr.val.clusterDim.x = attr.val.clusterDim.y = attr.val.clusterDim.z = 1;
  cudaLaunchConfig_t cfg{};
  cfg.blockDim = dim3(512);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = ctx->stream;
  cfg.attrs = &attr;
  cfg.numAttrs = 1;
  int parts = 1;
  for (int i = 0; i < 3 && (long long)T * (2 << i) <= ctx->sm_count; ++i) {
    if (ctx->chain_fit[i] < 0) {  // ~20 us a query; its shared memory allows one CTA per SM whatever M
      attr.val.clusterDim.x = 2 << i;
      cfg.gridDim = dim3(2u << i);
      if (cudaOccupancyMaxActiveClusters(&ctx->chain_fit[i], chain_kernel, &cfg) != cudaSuccess) {
        ctx->chain_fit[i] = 0;  // without an answer the smaller clusters do
        (void)cudaGetLastError();
      }
    }
    if (ctx->chain_fit[i] < (int)T) break;
    parts = 2 << i;
  }
  attr.val.clusterDim.x = parts;
  cfg.gridDim = dim3((unsigned)(T * parts));
  cudaLaunchKernelEx(&cfg, chain_kernel, (const ChainJob*)d_in, d_out);
  count_launch(ctx);
  std::vector<ChainOut> out(T);
  if ((e = check_cuda(ctx, cudaGetLastError(), "chain")) ||
      (e = check_cuda(ctx, cudaMemcpyAsync(out.data(), d_out, T * sizeof(ChainOut), cudaMemcpyDeviceToHost, ctx->stream),
                      "chain readback")) ||
      (e = stream_sync(ctx)))
    return e;
  const double seconds = std::chrono::duration<double>(std::chrono::steady_clock::now() - t0).count();
  long long total = 0;
  for (const ChainOut& o : out)
    for (int s = 0; s < 6; ++s) total += o.trees[s];
  for (size_t i = 0; i < T; ++i) {
    Trajectory* t = jobs[i];
    const ChainOut& o = out[i];
    for (int s = 0; s < o.steps; ++s) {
      const int k = t->M - 1 - (t->step + s);
      if (t->want_p0) t->p0[t->step + s] = o.p0[s];
      if ((o.clicked >> s) & 1u) t->S.push_back(k);
    }
    t->m = o.m;
    t->need_full = o.need_full;
    t->kappa_prev = o.kappa_prev;
    t->relD = o.relD;
    // a rejected attempt's last step is not counted as done (its state is dropped)
    t->step += o.code == kChainRejected ? o.steps - 1 : o.steps;
    if (o.code == kChainDone) t->state = Trajectory::kDone;
    if (o.code == kChainRejected) {
      t->state = Trajectory::kRejected;
      stt.rejections++;
    }
    t->host_step = o.code == kChainHost;
    stt.near_ties += o.near_ties;
    stt.uncertified += o.uncertified;
    for (int s = 0; s < 6; ++s) {
      stt.trees[s] += o.trees[s];
      stt.steps += o.trees[s];
      if (total > 0) stt.tree_seconds[s] += seconds * (double)o.trees[s] / (double)total;
    }
  }
  return GBS_OK;
}

}  // namespace gbs
