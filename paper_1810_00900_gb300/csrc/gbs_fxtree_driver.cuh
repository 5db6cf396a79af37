// Host side of the fixed-point tree engine: plan, workspace, launches.
#pragma once
#include <algorithm>
#include <string>
#include <vector>

#include "gbs_batch_driver.cuh"
#include "gbs_fxtree.cuh"

namespace gbs {

// Words of the matrices of level k of a tree over n modes (k = -1: the root), `count`
// matrices of it at a time.
inline long long fx_level_words(int n, int k, long long count, int L) {
  const int q = k < 0 ? n : n - 1 - k;
  if (k >= 5) count = (count + 31) / 32 * 32;
  return count * (long long)sym(2 * q) * L;
}

template <class E>
gbs_status fx_batch_run(gbs_ctx* ctx, int ntrees, const BatchTree* in, const void* roots_dev, int* status_dev,
                        const BatchTune& tune, const TreeFinish& fin) {
  typedef typename fx_sum<E>::type S;
  constexpr int L = sizeof(E) / 4;
  // Small trees (fx_small_kernel): one CTA for up to kOne modes, whose levels fit its
  // shared memory; up to 17 modes a CTA per setting of the first ones, as long as the
  // call's CTAs are few.  One launch of them against levels, us: 64 fraction bits, 32
  // trees of 12 .. 15 modes (~640 CTAs) 198 against 231, 4 of 17 (1024) 181 / 173; 128
  // bits, 8 of 15 (512) 168 / 201, 4 of 17 (1024) 320 / 221; 160 bits, 24 of 12 (384)
  // 182 / 210, 8 of 15 (1024) 268 / 215; 192 bits, one of 17 (512) 216 / 192.
  constexpr int LS = sizeof(S) / 4;
  constexpr int kOne = fx_small_words(10, 10, L, LS) * 4 <= 220 * 1024 ? 10 : 9;
  constexpr int kSub = kOne - 1;  // modes of a CTA's own tree where it is one of several
  long long ctas = 0;
  for (int i = 0; i < ntrees; ++i) {
    if (in[i].n < 1 || in[i].n > 32) return set_error(ctx, GBS_EINVAL, "batch tree size out of range");
    if (in[i].n > kOne) ctas += 1LL << std::min(in[i].n - kSub, 20);
  }
  const int small_max = ctas <= ctx->sm_count * (L <= 3 ? 6 : L <= 5 ? 4 : 2.5) ? 17 : kOne;
  std::vector<int> order;  // the others, largest first: every per-size list below is then a run of trees
  std::vector<FxSmall> small[2];  // in one CTA, in several
  int small_n[2] = {0, 0};
  long long blocks[2] = {0, 0};
  for (int i = 0; i < ntrees; ++i) {
    const int n = in[i].n, several = n > kOne ? 1 : 0;
    if (n > small_max) {
      order.push_back(i);
      continue;
    }
    const int d0 = several ? n - kSub : 0;
    small[several].push_back(FxSmall{blocks[several], in[i].root_off, fin.scale[i], n, d0, i, 0});
    blocks[several] += 1LL << d0;
    small_n[several] = std::max(small_n[several], n);
  }
  ntrees = (int)order.size();
  // the timer takes the leaf launches, or the small trees' where there are none
  cudaStream_t s = ctx->stream;
  auto timer = [&](bool stop) {
    if (!ctx->timing) return;
    KernelTimer& tm = ctx->fx_leaf_timer;
    if (!tm.start) {
      cudaEventCreate(&tm.start);
      cudaEventCreate(&tm.stop);
    }
    cudaEventRecord(stop ? tm.stop : tm.start, s);
    if (stop) tm.pending = true;
  };
  // Everything uploaded: what follows may go beside what the caller queues next.
  auto fork = [&]() -> gbs_status {
    if (!fin.beside) return GBS_OK;
    if (const gbs_status e = side_fork(ctx)) return e;
    s = ctx->side;
    return GBS_OK;
  };
  // Launched once the others' plan is known to fit: a batch that goes in parts by its plan has
  // not run its small trees yet.
  gbs_status st;
  auto launch_small = [&]() -> gbs_status {
    const void* d_small[2] = {};
    for (int c = 0; c < 2; ++c)
      if ((st = stage(ctx, small[c].data(), small[c].size() * sizeof(FxSmall), &d_small[c]))) return st;
    if ((st = dev_reserve(ctx, ctx->small_parts, (size_t)blocks[1] * sizeof(FxPart<S>)))) return st;
    if (ntrees == 0) {
      if ((st = fork())) return st;
      timer(false);
    }
    for (int c = 0; c < 2; ++c) {
      if (small[c].empty()) continue;
      const int smem = fx_small_words(small_n[c], c ? kSub : small_n[c], L, LS) * 4;
      if ((st = allow_smem(ctx, fx_small_kernel<E>, (size_t)smem, "small tree smem"))) return st;
      int threads = c || small_n[c] >= 8 ? 512 : small_n[c] >= 6 ? 256 : small_n[c] >= 4 ? 128 : 32;
      if (blocks[c] > ctx->sm_count) threads = std::min(threads, 256);  // two CTAs per SM
      fx_small_kernel<E><<<(unsigned)blocks[c], threads, smem, s>>>(
          (const FxSmall*)d_small[c], (int)small[c].size(), (const double*)roots_dev, fin.u, fin.extra,
          (FxPart<S>*)ctx->small_parts.ptr, fin.counts, status_dev, fin.po);
      count_launch(ctx);
      if ((st = check_cuda(ctx, cudaGetLastError(), "small trees"))) return st;
    }
    if (ntrees == 0) timer(true);
    return GBS_OK;
  };
  if (ntrees == 0) return launch_small();
  // ---------------- plan
  std::stable_sort(order.begin(), order.end(), [&](int a, int b) { return in[a].n > in[b].n; });
  // Levels per leaf thread.
  constexpr int kLeafQ = L <= 3 ? 3 : 2;
  const int Qmax = std::max(1, std::min(kLeafQ, 3 - tune.q_drop));
  const int nmax = in[order[0]].n;
  // Depth of the top kernel: at most tune.d_top and 256 CTAs, at least the five levels
  // that are not kept in tiles.  (A step of it against a level launch: N = 18 .. 20,
  // FP64, 171, 203, 233 us with 64 CTAs, 146, 176, 212 with 256, 160, 180, 216 with 1024.)
  int d_top = 5;
  while (d_top < tune.d_top && ((long long)ntrees << (d_top + 1)) <= 256) ++d_top;
  auto cta_smem = [&](int R, int TW) { return (size_t)((5 * L + 1) + R * (6 * L + 1)) * TW * 4; };
  std::vector<FxTree> trees(ntrees);
  std::vector<int> Q(ntrees);
  for (int i = 0; i < ntrees; ++i) {
    const BatchTree& b = in[order[i]];
    Q[i] = std::min(b.n, Qmax);
    trees[i] = FxTree{b.root_off, 0, fin.scale[order[i]], b.n, b.n - Q[i], order[i], 34 * i, 0, 0};
  }
  const int D0 = trees[0].D;
  // Workspace: all levels of all trees, and a partial sum per leaf CTA (N = 20, 24, 26, 28:
  // 63 MB, 1.0, 3.9, 15.6 GB with 64 fraction bits, 157 MB, 2.5, 9.8, 39 GB with 160).  A
  // single tree beyond its limit, a sixteenth of the device, goes in chunks of 2^cb nodes of
  // depth d0 (FxTree).  Where the device or the context's budget has less than the limit
  // left, a batch is evaluated in parts and a single tree in more chunks.
  // Tiles per warp: about five waves of the 16 warps an SM holds.  (One wave, and a few
  // CTAs more than that because every tree ends in a part of one, took twice its time:
  // 300 trees of 15 .. 17 modes, 64 fraction bits, 685 us.)
  auto tiles_of = [&](int i, int d0, int cb) { return ((1LL << (trees[i].D - d0 + cb)) + 31) / 32; };
  auto tpu_of = [&](int d0, int cb) {
    long long tiles = 0;
    for (int i = 0; i < ntrees; ++i) tiles += tiles_of(i, d0, cb);
    return (int)std::max(1LL, std::min(64LL, tiles / (80LL * ctx->sm_count)));
  };
  auto units_of = [&](int i, int d0, int cb, int tpu) { return (tiles_of(i, d0, cb) + 4 * tpu - 1) / (4 * tpu); };
  auto level_count = [](int k, int d0, int cb) { return d0 == 0 || k < d0 ? 1LL << k : 1LL << (k - d0 + cb); };
  auto s_count = [&](int i, int d0, int cb) {
    const int D = trees[i].D;
    return d0 ? (1LL << d0) + (1LL << (D - d0 + cb)) - (1LL << cb) : 1LL << D;
  };
  auto r32 = [](long long w) { return (w + 31) / 32 * 32; };
  auto r256 = [](size_t b) { return (b + 255) / 256 * 256; };
  struct Space {
    int d0, cb;
    size_t nodes, s, total;
  };
  auto space_of = [&](int d0, int cb) {
    const int tpu = tpu_of(d0, cb);
    long long words = 0, sv = 0, units = 0;
    for (int i = 0; i < ntrees; ++i) {
      const int n = trees[i].n;
      words += r32(fx_level_words(n, -1, 1, L));
      for (int k = 0; k < trees[i].D; ++k) words += r32(fx_level_words(n, k, level_count(k, d0, cb), L));
      sv += s_count(i, d0, cb);
      units += units_of(i, d0, cb, tpu) << (d0 - cb);
    }
    const size_t nodes = r256((size_t)words * 4), s = r256((size_t)sv * sizeof(S));
    return Space{d0, cb, nodes, s, nodes + s + (size_t)units * sizeof(FxPart<S>)};
  };
  // The fewest chunks that fit, from the deepest level on, since each chunk repeats the
  // launches below it (160 bits, N = 24 in 2 GB: 2.41 ms, 2.52 from the shallowest level on,
  // 2.37 whole; N = 26 in 8, 4, 1 GB 8.62, 8.84, 10.2 ms, 8.61 whole); the least there is where
  // nothing fits.
  auto fit = [&](size_t limit) {
    Space least = space_of(0, 0);
    if (least.total <= limit) return least;
    for (int chunk_bits = 1; chunk_bits <= D0 - 5; ++chunk_bits)  // log2 of the number of chunks
      for (int d = D0 - 1; d >= std::max(5 + chunk_bits, std::min(d_top, D0)); --d) {
        const Space c = space_of(d, d - chunk_bits);
        if (c.total <= limit) return c;
        if (c.total < least.total) least = c;
      }
    return least;
  };
  Space space = ntrees > 1 ? space_of(0, 0) : fit(ctx->tree_cap_bytes);
  if (ntrees > 1 && space.total > ctx->batch_cap_bytes) {
    ctx->batch_split = true;  // the caller evaluates the batch in parts
    return GBS_ENOMEM;
  }
  if ((st = launch_small())) return st;  // they run while a context's first call allocates
  // one allocation: a context's first call pays for each
  DevBuf& buf = fin.beside ? ctx->side_nodes : ctx->lvl[0];
  while ((st = dev_reserve(ctx, buf, space.total)) == GBS_ENOMEM) {
    if (ntrees > 1) {
      ctx->batch_split = true;
      return st;
    }
    const Space less = fit(space.total / 2);
    if (less.total >= space.total) return st;
    space = less;
  }
  if (st) return st;
  const int d0 = space.d0, cb = space.cb;
  std::vector<long long> off(34 * (size_t)ntrees, 0);
  long long words = 0, selems = 0;
  for (int i = 0; i < ntrees; ++i) {
    const int n = trees[i].n, D = trees[i].D;
    long long* o = &off[34 * (size_t)i];
    o[0] = words;
    words += r32(fx_level_words(n, -1, 1, L));
    for (int k = 0; k < D; ++k) {
      o[k + 1] = words;
      words += r32(fx_level_words(n, k, level_count(k, d0, cb), L));
    }
    trees[i].s_base = selems;
    selems += s_count(i, d0, cb);
  }
  const int chunks = 1 << (d0 - cb);
  std::vector<FxTree> chunked = trees;
  for (FxTree& t : chunked) t.d0 = d0, t.cb = cb;
  // top: the levels below min(D, d_top)
  std::vector<FxSeg> top(ntrees);
  long long top_blocks = 0;
  auto dtop_of = [&](int i) { return std::min(trees[i].D, d_top); };
  for (int i = 0; i < ntrees; ++i) {
    top[i] = FxSeg{top_blocks, i, 0};
    top_blocks += 1LL << dtop_of(i);
  }
  // levels, by child size q downwards
  struct Launch {
    int q, TW, W;  // TW = 0: a warp per 32 children; else W warps per TW children
    std::vector<FxSeg> segs;
    long long children, blocks;
    size_t at, smem;
    bool in_chunk;
  };
  std::vector<Launch> levels;
  for (int q = nmax - 1; q >= 1; --q) {
    Launch l{q, 0, 1, {}, 0, 0, 0, 0, false};
    for (int i = 0; i < ntrees; ++i) {
      const int k = trees[i].n - 1 - q;
      if (k < dtop_of(i) || k >= trees[i].D) continue;
      l.in_chunk = d0 > 0 && k >= d0;
      l.segs.push_back(FxSeg{l.children, i, 0});
      l.children += 1LL << (l.in_chunk ? k - d0 + cb : k);
    }
    if (l.segs.empty()) continue;
    const int R = 2 * q;
    const long long tiles = l.children / 32;
    if (tiles >= 8LL * ctx->sm_count && q <= 5) {
      l.smem = (size_t)3 * R * L * 128;
    } else {
      // CTAs of 4 warps for 16 children; where that is too few, more warps for fewer
      l.TW = 16;
      while (l.TW > 1 && l.children / l.TW < ctx->sm_count) l.TW /= 2;
      l.W = l.children / l.TW < 3LL * ctx->sm_count ? 8 : 4;
      while (l.W > 1 && 32 / l.TW * l.W > std::max(R, sym(R) / 2)) l.W /= 2;
      l.smem = cta_smem(R, l.TW);
    }
    const int per = l.TW ? l.TW : 32;
    for (FxSeg& sg : l.segs) sg.first /= per;
    l.blocks = l.children / per;
    levels.push_back(l);
  }
  // leaves, one launch per Q
  struct Leaf {
    int Q;
    std::vector<FxSeg> segs;
    long long units;
    size_t at;
  };
  std::vector<Leaf> leaves;
  std::vector<FxSeg> sums;
  long long units_total = 0;
  const int tpu = tpu_of(d0, cb);
  for (int i = 0; i < ntrees; ++i) {
    if (leaves.empty() || leaves.back().Q != Q[i]) leaves.push_back(Leaf{Q[i], {}, 0, 0});
    Leaf& lf = leaves.back();
    const long long units = units_of(i, d0, cb, tpu);
    lf.segs.push_back(FxSeg{lf.units, i, tpu});
    lf.units += units;
    sums.push_back(FxSeg{units_total, i, 0});
    units_total += units * chunks;
  }
  sums.push_back(FxSeg{units_total, 0, 0});
  // ---------------- upload
  Blob blob;
  const size_t o_trees = blob.put(trees), o_chunked = blob.put(chunked), o_off = blob.put(off), o_top = blob.put(top);
  for (Launch& l : levels) l.at = blob.put(l.segs);
  for (Leaf& l : leaves) l.at = blob.put(l.segs);
  const size_t o_sums = blob.put(sums);
  const unsigned char* plan = nullptr;
  if ((st = stage(ctx, blob.bytes.data(), blob.bytes.size(), (const void**)&plan))) return st;
  uint32_t* nodes = (uint32_t*)buf.ptr;
  S* sval = (S*)((unsigned char*)nodes + space.nodes);
  FxPart<S>* parts = (FxPart<S>*)((unsigned char*)nodes + space.nodes + space.s);
  const FxTree* d_trees = (const FxTree*)(plan + o_trees);
  const FxTree* d_chunked = (const FxTree*)(plan + o_chunked);
  const long long* d_off = (const long long*)(plan + o_off);

  // ---------------- launches
  const int smem_top = sym(2 * nmax) * (int)sizeof(E) + 2 * nmax * (int)sizeof(FxRow<E>);
  size_t smem_cta = 0;
  for (const Launch& l : levels)
    if (l.TW) smem_cta = std::max(smem_cta, l.smem);
  if ((st = allow_smem(ctx, fx_top_kernel<E>, (size_t)smem_top, "top smem")) ||
      (st = allow_smem(ctx, fx_level_cta_kernel<E>, smem_cta, "level smem")))
    return st;
  if ((st = fork())) return st;
  fx_top_kernel<E><<<(unsigned)top_blocks, 256, smem_top, s>>>((const FxSeg*)(plan + o_top), ntrees, d_trees, d_off,
                                                               (const double*)roots_dev, nodes, sval, status_dev);
  count_launch(ctx);
  long long before = top_blocks;  // CTAs of the launch before
  auto early = [&](long long blocks) {
    const bool e = before <= 2LL * ctx->sm_count;
    before = blocks;
    return e;
  };
  auto level = [&](const Launch& l, unsigned chunk) {
    const bool el = early(l.blocks);
    const FxSeg* sg = (const FxSeg*)(plan + l.at);
    const int ns = (int)l.segs.size();
    const FxTree* tr = l.in_chunk ? d_chunked : d_trees;
    if (l.TW)
      launch_early(el, fx_level_cta_kernel<E>, (unsigned)l.blocks, 32 * l.W, l.smem, s, sg, ns, tr, d_off, l.q, l.TW, chunk, nodes,
                sval, status_dev);
    else if (l.q >= 4)
      launch_early(el, fx_level_warp_kernel<E, 4>, (unsigned)l.blocks, 32, l.smem, s, sg, ns, tr, d_off, l.q, chunk, nodes, sval,
                status_dev);
    else
      launch_early(el, fx_level_warp_kernel<E, 2>, (unsigned)l.blocks, 32, l.smem, s, sg, ns, tr, d_off, l.q, chunk, nodes, sval,
                status_dev);
    count_launch(ctx);
  };
  for (const Launch& l : levels)
    if (!l.in_chunk) level(l, 0u);
  timer(false);
  for (int h = 0; h < chunks; ++h) {
    for (const Launch& l : levels)
      if (l.in_chunk) level(l, (unsigned)h);
    long long base = h * leaves[0].units;  // chunks: one tree, one leaf launch each
    for (const Leaf& l : leaves) {
      const unsigned grid = (unsigned)l.units;
      const FxSeg* sg = (const FxSeg*)(plan + l.at);
      const int ns = (int)l.segs.size();
      const bool el = early(grid);
      switch (l.Q) {
        case 1: launch_early(el, fx_leaf_kernel<E, 1>, grid, 128, 0, s, sg, ns, (unsigned)h, d_chunked, d_off, nodes, sval, parts + base, status_dev); break;
        case 2: launch_early(el, fx_leaf_kernel<E, 2>, grid, 128, 0, s, sg, ns, (unsigned)h, d_chunked, d_off, nodes, sval, parts + base, status_dev); break;
        default: launch_early(el, fx_leaf_kernel<E, kLeafQ>, grid, 128, 0, s, sg, ns, (unsigned)h, d_chunked, d_off, nodes, sval, parts + base, status_dev); break;
      }
      count_launch(ctx);
      base += l.units;
    }
  }
  timer(true);
  const int final_threads = units_total > 256LL * ntrees ? 1024 : 128;
  launch_early(early(0), fx_final_kernel<S>, (unsigned)ntrees, final_threads, 0, s, parts, (const FxSeg*)(plan + o_sums), d_trees,
            status_dev, fin.u, fin.extra, fin.po);
  count_launch(ctx);
  return check_cuda(ctx, cudaGetLastError(), "fixed-point batch launch");
}

}  // namespace gbs
