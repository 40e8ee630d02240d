// su3_f64_meas.cu -- what measures SU(3) FP64 lattices: the overrelaxation kernels of a
// working sweep's last pass that also sum plaquettes, and the measurement of a
// configuration.
#include "qcd_su3d.cuh"

namespace qcd {
cudaError_t su3d_launch_or_meas(const Ctx& a, int parity, int mu, cudaStream_t st) {
  return su3d_launch_level<KIND_OR_MEAS>(a, parity, mu, st);
}

namespace {
template <int FIELD>
__device__ __noinline__ double2 plaquettes_fp64(const Ctx& a, int64_t idx) {
  SumD v0, v1;
  plaquette_site<SU3Policy<double>, FIELD>(a, idx, v0, v1);
  return make_double2(v0.s, v1.s);
}

// Plaquettes of 32 sites (parity p, indices base ..): Re Tr of (Ut_mu(x) Ut_nu(x+mu))
// (Ut_nu(x) Ut_mu(x+nu))^+, row by row; the warp's spatial and temporal sums.
template <int FIELD>
__device__ __forceinline__ void su3d_plaquettes(const Ctx& a, int p, int base, Su3dMeasTiles& sh, int role, int lane,
                                                int bar, double& v0, double& v1) {
  const int h = min(base + lane, a.g.Vh - 1);
  const bool in = base + lane < a.g.Vh;
  const Site x = site_of(a.g, p, h);
  const int s0 = lex(a.g, x);
  const double2* links = reinterpret_cast<const double2*>(a.links);
  auto link = [&](int m, int q, int s) { return links + (m * 2 + q) * a.g.plane + (s >> 1); };
  auto ahead = [&](int d) {
    const int c = d == 0 ? x.x : d == 1 ? x.y : d == 2 ? x.z : x.t, ext = d == 3 ? a.g.Nt : a.g.Ns;
    const int st = d == 0 ? 1 : d == 1 ? a.g.Ns : d == 2 ? a.g.Ns * a.g.Ns : a.g.Ns * a.g.Ns * a.g.Ns;
    return c == ext - 1 ? st - ext * st : st;
  };
  uint32_t big = 0, bad = 0;
  int64_t sum[2] = {0, 0};
#pragma unroll 1
  for (int q = 0; q < 6; ++q) {
    const int mu = q < 3 ? 0 : q < 5 ? 1 : 2, nu = q < 3 ? q + 1 : q < 5 ? q - 1 : 3;
    FxC u[3], w[3], ab[3];
    // rows of Ut_nu(x+mu) and Ut_mu(x+nu) for the three warps
    const RawRow r0 = su3d_row(a, link(nu, p ^ 1, s0 + ahead(mu)), role, false);
    const RawRow r1 = su3d_row(a, link(mu, p ^ 1, s0 + ahead(nu)), role, false);
    su3d_convert<1>(r0, false, u, big);
    su3d_convert<1>(r1, false, w, big);
    if (FIELD && nu == 1) su3d_scale<FIELD, false>(a, mu == 0 ? x.x + ahead(0) : x.x, u, bad);
    if (FIELD && mu == 1) su3d_scale<FIELD, false>(a, x.x, w, bad);
    if (q > 0) bar_96(bar);  // the tiles' readers are done
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      sh.t[0][role][k].put(lane, u[k]);
      sh.t[1][role][k].put(lane, w[k]);
    }
    su3d_convert<0>(su3d_row(a, link(mu, p, s0), role, false), false, u, big);
    su3d_convert<0>(su3d_row(a, link(nu, p, s0), role, false), false, w, big);
    if (FIELD && mu == 1) su3d_scale<FIELD, false>(a, x.x, u, bad);
    if (FIELD && nu == 1) su3d_scale<FIELD, false>(a, x.x, w, bad);
    bar_96(bar);
#pragma unroll
    for (int j = 0; j < 3; ++j) {
      FxDot<false> d;
#pragma unroll
      for (int k = 0; k < 3; ++k) d.add(u[k], sh.t[0][k][j].get(lane));
      ab[j] = d.limbs(bad);
    }
    uint32_t parts = 0;
#pragma unroll
    for (int j = 0; j < 3; ++j) parts |= fx_part(ab[j].re) | fx_part(ab[j].im);
    if (fx_tiny(parts)) bad |= FX_BAD;
    FxAcc t;
#pragma unroll
    for (int j = 0; j < 3; ++j) {
      FxDot<false> d;
#pragma unroll
      for (int k = 0; k < 3; ++k) d.add(w[k], sh.t[1][k][j].get(lane));
      const FxC dc = d.limbs(bad);
      t.add(ab[j].re, dc.re);
      t.add(ab[j].im, dc.im);
    }
    const int64_t v = t.value();
    fx_check(v, bad);
    sum[nu == 3] += v;
  }
  sh.flag[role][lane] = (bad & FX_BAD) | (big & FX_BIG);
  bar_96(bar);
  const bool out_of_range = sh.flag[0][lane] | sh.flag[1][lane] | sh.flag[2][lane];
  v0 = fx_warp_sum(in && !out_of_range ? sum[0] : 0);
  v1 = fx_warp_sum(in && !out_of_range ? sum[1] : 0);
  if (role == 0 && __any_sync(0xffffffffu, in && out_of_range)) {
    SumD w0, w1;
    if (in && out_of_range) {
      const double2 v = plaquettes_fp64<FIELD>(a, int64_t(p) * a.g.Vh + h);
      w0.s = v.x;
      w1.s = v.y;
    }
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) {
      w0.merge_down(off);
      w1.merge_down(off);
    }
    v0 += 3.0 * w0.s;  // plaquette_site takes the 1/3
    v1 += 3.0 * w1.s;
  }
}

// Measurement of a configuration: CTAs of eight groups of three warps, 256 sites (as
// measure_kernel's blocks, for the same partials): plaquettes, then the Polyakov loop.
// Measurement at 16^3x4 / 32^3x8 / 48^3x16, us: 60 / 344 / 2200, against 128 / 772 /
// 4880 by the FP64 kernel (SU(2), one thread a site: 23 / 66 / 394 against 42 / 159 / 898).
template <int FIELD>
__global__ void __launch_bounds__(768) su3d_measure_kernel(const __grid_constant__ Ctx a, int n_plaq_blocks) {
  extern __shared__ __align__(16) unsigned char smem[];
  Su3dMeasTiles* tiles = reinterpret_cast<Su3dMeasTiles*>(smem);
  __shared__ double sum[24][2];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, group = warp / 3, role = warp - 3 * group;
  double v0 = 0.0, v1 = 0.0;
  if (int(blockIdx.x) < n_plaq_blocks) {  // groups of either parity by turns
    const int base = (blockIdx.x * 4 + (group >> 1)) * 32;
    if (base < a.g.Vh) su3d_plaquettes<FIELD>(a, group & 1, base, tiles[group], role, lane, 1 + group, v0, v1);
  } else {
    const int base = ((int(blockIdx.x) - n_plaq_blocks) * 8 + group) * 32;
    if (base < a.g.Ns * a.g.Ns * a.g.Ns) su3d_poly(a, base, tiles[group], role, lane, 1 + group, v0, v1);
  }
  if (lane == 0) {
    sum[warp][0] = v0;
    sum[warp][1] = v1;
  }
  __syncthreads();
  if (warp == 0) {  // a tree: 5 roundings on a path and 5 FP64 instructions instead of 23
    const int g = 3 * ((lane >> 1) & 7), k = lane & 1;
    double r = sum[g][k] + sum[g + 1][k] + sum[g + 2][k];
#pragma unroll
    for (int off = 8; off > 1; off >>= 1) r += __shfl_down_sync(0xffffffffu, r, off);
    if (lane < 2) a.partials[2 * int64_t(blockIdx.x) + lane] = r;
  }
}

template <int FIELD>
inline cudaError_t su3d_launch_measure_field(const Ctx& a, cudaStream_t st) {
  constexpr int bytes = 8 * int(sizeof(Su3dMeasTiles));
  const cudaError_t e =
      cudaFuncSetAttribute(su3d_measure_kernel<FIELD>, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
  if (e != cudaSuccess) return e;
  const int np = meas_plaq_blocks(a.g), nl = meas_poly_blocks(a.g);
  su3d_measure_kernel<FIELD><<<np + nl, 768, bytes, st>>>(a, np);
  launch_measure_final(a, st, np, nl, 3.0, 3.0);
  return cudaGetLastError();
}

}  // namespace

cudaError_t su3d_launch_measure(const Ctx& a, int effective, cudaStream_t st) {
  switch (effective ? su3_field_level(a) : 0) {
    case 0: return su3d_launch_measure_field<0>(a, st);
    case 1: return su3d_launch_measure_field<1>(a, st);
    default: return su3d_launch_measure_field<2>(a, st);
  }
}
}  // namespace qcd
