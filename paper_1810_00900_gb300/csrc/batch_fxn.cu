// Batched subset-determinant trees, narrow fixed-point per-term arithmetic
// (128 fraction bits, real basis).
#include "gbs_fxtree_driver.cuh"

namespace gbs {
gbs_status batch_fxn_real(gbs_ctx* ctx, int ntrees, const BatchTree* trees, const void* roots, int* status,
                         const BatchTune& tune, const TreeFinish& fin) {
  return fx_batch_run<fxn4>(ctx, ntrees, trees, roots, status, tune, fin);
}
}  // namespace gbs
