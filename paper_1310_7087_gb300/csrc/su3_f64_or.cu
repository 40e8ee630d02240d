// su3_f64_or.cu -- the SU(3) FP64 overrelaxation kernels that also reunitarize each
// link they update (the last pass of a sweep).
#include "qcd_su3d.cuh"

namespace qcd {
cudaError_t su3d_launch_or_reunit(const Ctx& a, int parity, int mu, cudaStream_t st) {
  return su3d_launch_level<KIND_OR_REUNIT>(a, parity, mu, st);
}
}  // namespace qcd
