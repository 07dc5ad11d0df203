// F64 instantiation of the phase-B kernels; a translation unit of its own, so that the
// phases build in parallel.
#include "dg_aux.h"
#include "dg_launch.cuh"

namespace dgnn {
cudaError_t surface_f64(const dg_ctx* c, double* q, double* dqdt, const Forcing& f, int mode, const RkStage& rk,
                       double dt, cudaStream_t st) {
  return surface_t<double>(c, q, dqdt, f, mode, rk, dt, st);
}
}  // namespace dgnn
