// su3_f64.cu -- kernels of the gauge sweep for SU(3) with FP64 18-real links.
// The phase update and the measurements use the fixed-point kernels of
// qcd_su3d.cuh and su3_f64_meas.cu; reunitarization, start and layout conversion use
// the shared templates.
#include "qcd_su3d.cuh"

namespace qcd {
namespace {
cudaError_t launch_phase(const Ctx& a, int kind, int parity, int mu, int /*block: the kernel's own*/,
                         cudaStream_t st) {
  if (kind == KIND_HB) return su3d_launch_hb(a, parity, mu, st);
  if (kind == KIND_OR) return su3d_launch_level<KIND_OR>(a, parity, mu, st);
  if (kind == KIND_OR_MEAS && mu >= 1) return su3d_launch_or_meas(a, parity, mu, st);
  return su3d_launch_or_reunit(a, parity, mu, st);
}

// Block sizes that qcd_set_block takes (those of the 96-register FP64 kernel
// that this storage had; the CTA shape is part of the kernel now).
int max_phase_block() { return 640; }
bool own_shape(const GeomH&) { return true; }
}  // namespace

using SU3D = SU3Policy<double>;
const PolicyOps kOpsSU3F64 = PolicyOps{3,
                                       0,
                                       SU3D::COMPS,
                                       &launch_phase,
                                       &launch_reunit<SU3D>,
                                       &launch_start<SU3D>,
                                       &su3d_launch_measure,
                                       &launch_to_canonical<SU3D>,
                                       &launch_from_canonical<SU3D>,
                                       &launch_set_frozen<SU3D>,
                                       &su3d_measure_fused_tail,
                                       &max_phase_block,
                                       &own_shape};
}  // namespace qcd
