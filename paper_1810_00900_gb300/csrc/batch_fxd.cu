// Batched subset-determinant trees, FP64 precision on the integer pipe (64 fraction
// bits, real basis) for states that bound the tree.
#include "gbs_fxtree_driver.cuh"

namespace gbs {
gbs_status batch_fxd_real(gbs_ctx* ctx, int ntrees, const BatchTree* trees, const void* roots, int* status,
                          const BatchTune& tune, const TreeFinish& fin) {
  return fx_batch_run<fxd>(ctx, ntrees, trees, roots, status, tune, fin);
}
}  // namespace gbs
