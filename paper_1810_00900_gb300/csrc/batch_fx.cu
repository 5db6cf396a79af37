// Batched subset-determinant trees, fixed-point (160 fraction bits) per-term arithmetic (real basis).
#include "gbs_fxtree_driver.cuh"

namespace gbs {
gbs_status batch_fx_real(gbs_ctx* ctx, int ntrees, const BatchTree* trees, const void* roots, int* status,
                         const BatchTune& tune, const TreeFinish& fin) {
  return fx_batch_run<fx>(ctx, ntrees, trees, roots, status, tune, fin);
}
}  // namespace gbs
