// su3_f64_hb.cu -- the SU(3) FP64 heat-bath kernels, in a translation unit of their
// own so they compile in parallel with su3_f64.cu.
#include "qcd_su3d.cuh"

namespace qcd {
cudaError_t su3d_launch_hb(const Ctx& a, int parity, int mu, cudaStream_t st) {
  return su3d_launch_level<KIND_HB>(a, parity, mu, st);
}
}  // namespace qcd
