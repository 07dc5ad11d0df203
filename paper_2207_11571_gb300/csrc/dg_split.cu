// Split-form phase A (kinetic-energy-preserving volume term) in both precisions: a
// translation unit of its own, so that these instantiations build in parallel with the
// default kernels.
#include "dg_aux.h"
#include "dg_launch.cuh"

namespace dgnn {
cudaError_t volume_split_f32(const dg_ctx* c, const double* q, int src, cudaStream_t st) {
  return volume_t<float, true>(c, q, src, st);
}
cudaError_t volume_split_f64(const dg_ctx* c, const double* q, int src, cudaStream_t st) {
  return volume_t<double, true>(c, q, src, st);
}
// Constant-memory tables of this unit's kernels (see upload_const_D).
cudaError_t prepare_split_constants() { return upload_const_D(); }
}  // namespace dgnn
