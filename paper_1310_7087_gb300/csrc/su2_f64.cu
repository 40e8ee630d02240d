// su2_f64.cu -- kernels of the gauge sweep for SU(2) with FP64 4-real links
// (quaternions).  The phase update uses the fixed-point kernels of
// qcd_su2d.cuh; reunitarization, start, measurements and layout conversion use
// the shared templates.
#include "qcd_su2d.cuh"

namespace qcd {
namespace {
cudaError_t launch_phase(const Ctx& a, int kind, int parity, int mu, int block, cudaStream_t st) {
  if (kind == KIND_HB) return su2d_launch_level<KIND_HB>(a, parity, mu, block, st);
  if (kind == KIND_OR) return su2d_launch_level<KIND_OR>(a, parity, mu, block, st);
  if (kind == KIND_OR_MEAS && mu >= 1) return su2d_launch_level<KIND_OR_MEAS>(a, parity, mu, block, st);
  return su2d_launch_level<KIND_OR_REUNIT>(a, parity, mu, block, st);
}

cudaError_t measure_fused_tail(const Ctx& a, int block, cudaStream_t st) {
  return su2c_measure_fused_tail<double>(a, su2d_links_per_cta(a.g, block), st);
}

int max_phase_block() { return 512; }  // the kernels' launch bound
}  // namespace

using SU2D = SU2Policy<double>;
const PolicyOps kOpsSU2F64 = PolicyOps{2,
                                       0,
                                       SU2D::COMPS,
                                       &launch_phase,
                                       &launch_reunit<SU2D>,
                                       &launch_start<SU2D>,
                                       &launch_measure<SU2D>,
                                       &launch_to_canonical<SU2D>,
                                       &launch_from_canonical<SU2D>,
                                       &launch_set_frozen<SU2D>,
                                       &measure_fused_tail,
                                       &max_phase_block};
}  // namespace qcd
