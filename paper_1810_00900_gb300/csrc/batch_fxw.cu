// Batched subset-determinant trees, wide fixed-point per-term arithmetic (real basis).
#include "gbs_fxtree_driver.cuh"

namespace gbs {
gbs_status batch_fxw_real(gbs_ctx* ctx, int ntrees, const BatchTree* trees, const void* roots, int* status,
                         const BatchTune& tune, const TreeFinish& fin) {
  return fx_batch_run<fxw>(ctx, ntrees, trees, roots, status, tune, fin);
}
}  // namespace gbs
