// F64 instantiation of the phase-A kernels.
#include "dg_aux.h"
#include "dg_launch.cuh"

namespace dgnn {
cudaError_t volume_f64(const dg_ctx* c, const double* q, int src, cudaStream_t st) {
  return volume_t<double, false>(c, q, src, st);
}
}  // namespace dgnn
