// Batched subset-determinant trees, td per-term arithmetic (real and complex).
#include "gbs_batch_driver.cuh"

namespace gbs {
gbs_status batch_td_real(gbs_ctx* ctx, int ntrees, const BatchTree* trees, const void* roots, int* status,
                          const BatchTune& tune, const TreeFinish& fin) {
  return batch_run<td, 3>(ctx, ntrees, trees, roots, status, tune, fin);
}
gbs_status batch_td_cplx(gbs_ctx* ctx, int ntrees, const BatchTree* trees, const void* roots, int* status,
                          const BatchTune& tune, const TreeFinish& fin) {
  return batch_run<cplx<td>, 2>(ctx, ntrees, trees, roots, status, tune, fin);
}
}  // namespace gbs
