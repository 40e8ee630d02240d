// su3_f32_hb.cu -- the SU(3) FP32 heat-bath kernels, in a translation unit of their
// own so they compile in parallel with su3_f32.cu.
#include "qcd_su3c.cuh"

namespace qcd {
cudaError_t su3c_launch_hb(const Ctx& a, int parity, int mu, int block, cudaStream_t st) {
  su3c_launch_level<KIND_HB>(a, parity, mu, block, st);
  return cudaGetLastError();
}

int su3c_hb_max_block() { return su3c_block_limit_level<KIND_HB>(); }
}  // namespace qcd
