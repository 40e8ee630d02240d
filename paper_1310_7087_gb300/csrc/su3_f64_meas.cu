// su3_f64_meas.cu -- the SU(3) FP64 overrelaxation kernels of a working sweep's last
// pass that also sum plaquettes.
#include "qcd_su3d.cuh"

namespace qcd {
cudaError_t su3d_launch_or_meas(const Ctx& a, int parity, int mu, cudaStream_t st) {
  return su3d_launch_level<KIND_OR_MEAS>(a, parity, mu, st);
}
}  // namespace qcd
