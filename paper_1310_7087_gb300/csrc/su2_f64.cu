// su2_f64.cu -- kernels of the gauge sweep for SU(2) with FP64 4-real links
// (quaternions).  The phase update uses the fixed-point kernels of
// qcd_su2d.cuh, the measurement is below; reunitarization, start and layout
// conversion use the shared templates.
#include "qcd_su2d.cuh"

namespace qcd {
namespace {
// Plaquettes of site x of parity p: (1/2) Re Tr of each by quaternions in fixed point;
// *v the spatial and temporal sums in FP64.
template <bool FIELD>
__device__ __forceinline__ void su2d_plaquettes(const Ctx& a, int p, int h, SumD (&v)[2]) {
  const LexSite x = lex_site(a, p, h);
  const int stride[4] = {1, a.g.Ns, a.g.Ns * a.g.Ns, a.g.Ns * a.g.Ns * a.g.Ns};
  uint32_t big = 0, bad = 0;
  int64_t sum[2] = {0, 0};
#pragma unroll
  for (int mu = 0; mu < 3; ++mu)
#pragma unroll
    for (int nu = mu + 1; nu < 4; ++nu) {
      auto ahead = [&](int d) {
        const int ext = d == 3 ? a.g.Nt : a.g.Ns;
        return x.c[d] == ext - 1 ? stride[d] - ext * stride[d] : stride[d];
      };
      Fx u[4], w[4], ab[4];
      int64_t t[4];
      auto load = [&](int d, int q, int s, int xc, Fx (&l)[4]) {
        su2d_load<false, false>(a, d, q, s, l, big);
        if (FIELD && d == 1) su2d_phase<false, false>(a, xc, l, bad);
      };
      load(mu, p, x.s, x.c[0], u);
      load(nu, p ^ 1, x.s + ahead(mu), mu == 0 ? x.c[0] + ahead(0) : x.c[0], w);
      fx_qmul(u, w, t);
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        fx_check(t[k], bad);
        ab[k] = fx_limbs(t[k]);
      }
      if (fx_tiny(fx_part(ab[0]) | fx_part(ab[1]) | fx_part(ab[2]) | fx_part(ab[3]))) bad |= FX_BAD;
      load(nu, p, x.s, x.c[0], u);
      load(mu, p ^ 1, x.s + ahead(nu), x.c[0], w);
      fx_qmul(u, w, t);
      FxAcc r;
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        fx_check(t[k], bad);
        r.add(ab[k], fx_limbs(t[k]));
      }
      const int64_t e = r.value();
      fx_check(e, bad);
      sum[nu == 3] += e;
    }
  if ((bad & FX_BAD) || (big & FX_BIG)) {
    plaquette_site<SU2Policy<double>, FIELD ? 1 : 0>(a, int64_t(p) * a.g.Vh + h, v[0], v[1]);
  } else {
    v[0].s = fx_double(sum[0]);
    v[1].s = fx_double(sum[1]);
  }
}

// As measure_kernel; the Polyakov loop (one product a site and time slice) stays FP64.
template <bool FIELD>
__global__ void __launch_bounds__(MEAS_THREADS, 2) su2d_measure_kernel(const __grid_constant__ Ctx a, int n_plaq_blocks) {
  SumD v[2];
  if (int(blockIdx.x) < n_plaq_blocks) {
    const int64_t idx = int64_t(blockIdx.x) * MEAS_THREADS + threadIdx.x;
    if (idx < 2LL * a.g.Vh) su2d_plaquettes<FIELD>(a, idx >= a.g.Vh, int(idx >= a.g.Vh ? idx - a.g.Vh : idx), v);
  } else {
    const int64_t idx = int64_t(int(blockIdx.x) - n_plaq_blocks) * MEAS_THREADS + threadIdx.x;
    if (idx < int64_t(a.g.Ns) * a.g.Ns * a.g.Ns) polyakov_site<SU2Policy<double>>(a, idx, v[0], v[1]);
  }
  block_sums(v, a.partials + 2 * blockIdx.x);
}

cudaError_t launch_measure_f64(const Ctx& a, int effective, cudaStream_t st) {
  const int np = meas_plaq_blocks(a.g), nl = meas_poly_blocks(a.g);
  if (effective && phases_on_links(a)) su2d_measure_kernel<true><<<np + nl, MEAS_THREADS, 0, st>>>(a, np);
  else su2d_measure_kernel<false><<<np + nl, MEAS_THREADS, 0, st>>>(a, np);
  launch_measure_final(a, st, np, nl, 1.0, 1.0);
  return cudaGetLastError();
}

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
                                       &launch_measure_f64,
                                       &launch_to_canonical<SU2D>,
                                       &launch_from_canonical<SU2D>,
                                       &launch_set_frozen<SU2D>,
                                       &measure_fused_tail,
                                       &max_phase_block,
                                       &su2d_split};
}  // namespace qcd
