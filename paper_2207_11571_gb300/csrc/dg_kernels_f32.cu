// F32 instantiation of the phase-A kernels.
#include "dg_aux.h"
#include "dg_launch.cuh"

namespace dgnn {
cudaError_t volume_f32(const dg_ctx* c, const double* q, int src, cudaStream_t st) {
  return volume_t<float, false>(c, q, src, st);
}
cudaError_t state_f32(const dg_ctx* c, const double* q, bool* done, cudaStream_t st) {
  return state_t<float>(c, q, done, st);
}
// Constant-memory tables of this unit's kernels (see upload_const_D).
cudaError_t prepare_f32_constants() { return upload_const_D(); }
}  // namespace dgnn
