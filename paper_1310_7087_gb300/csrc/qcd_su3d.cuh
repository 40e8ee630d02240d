// qcd_su3d.cuh -- phase kernel for SU(3) with FP64 links, its matrix products in
// fixed point (qcd_fix.cuh) on the integer pipe.
//
// Three warps share 32 links (lane = link).  Of a product X Y^+ Z^+ of three
// links, row i of the result needs row i of X and all of Y and Z, so warp i
// converts row i of each to fixed point, leaves Y's and Z's in shared memory and
// computes row i: no conversion is done twice, a thread holds rows instead of
// matrices (5 to 7 CTAs of 96 threads stay resident where one thread per link
// needs 168 registers), and the chain of one update is a third as long.  The
// update itself goes by columns: the subgroup rotations mix rows, so warp c
// rotates column c; the three rotations are found by one warp each.
//
// Bound: the integer pipes (ncu at 32^3x8: widening multiply-adds and moves keep
// the multiplier's pipe 61 % busy, adds, shifts and logic the ALU 51 %; 21,200
// warp instructions per 32 updates; fixed-latency waits and the pipes' are the
// largest stalls) where the FP64 form was bound by the FP64 unit (94 % busy).
// Overrelaxation / heat-bath phase of y-links, us, FP64 form -> this: 4^3x4 73.8 / 118.9
// -> 12 / 16.5; 16^3x4 75.8 / 126.2 -> 18.5 / 25; 32^3x8 447 / 710 -> 151 / 214;
// 48^3x16 2868 / 4314 -> 939 / 1408.  One thread per link (168 registers) took 1231 us
// for the overrelaxation of the last, with the matrices unrolled for both kinds of
// staple 1665 (instruction cache); applying the rotations to the rows by one copy of
// the code for all three subgroups (finding them is one copy) 1 to 2 % more.
#pragma once

#include <type_traits>

#include "qcd_fixmath.cuh"
#include "qcd_kernels.cuh"

namespace qcd {

// Row r of a link, or of its adjoint (dag), as stored; the imaginary parts of
// the adjoint still want their sign.
struct RawRow {
  double2 v[3];
};
__device__ __forceinline__ RawRow su3d_row(const Ctx& a, const double2* p, int r, bool dag) {
  const int64_t stride = 8 * a.g.plane;
  p += r * (dag ? stride : 3 * stride);
  const int64_t step = dag ? 3 * stride : stride;
  return {{__ldg(p), __ldg(p + step), __ldg(p + 2 * step)}};
}
template <int INT>
__device__ __forceinline__ Fx su3d_fx(double x, uint32_t& big) {
  return INT ? fx_load_int(x, big) : fx_load(x, big);
}
template <int INT>
__device__ __forceinline__ void su3d_convert(const RawRow& w, bool dag, FxC r[3], uint32_t& big) {
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    const int flip = dag ? int(0x80000000u) : 0;
    r[k] = {su3d_fx<INT>(w.v[k].x, big),
            su3d_fx<INT>(__hiloint2double(__double2hiint(w.v[k].y) ^ flip, __double2loint(w.v[k].y)), big)};
  }
}

// Factor k of the diagonal y-link background at x (lambda3 alone: factor 2 is 1
// and callers leave it out).
template <int FIELD>
__device__ __forceinline__ FxC su3d_b(const Ctx& a, int x, int k) {
  uint32_t e = 0;
  const double2 v = FIELD == 1 ? __ldg(a.phase64 + x) : __ldg(a.phase64 + a.g.Ns + 3 * x + k);
  return {fx_load_int(v.x, e), fx_load_int(FIELD == 1 && k == 1 ? -v.y : v.y, e)};
}
// v_k <- v_k b_k, CONJ: conj(b_k)
template <int FIELD, bool CONJ>
__device__ __forceinline__ void su3d_scale(const Ctx& a, int x, FxC v[3], uint32_t& bad) {
#pragma unroll
  for (int k = 0; k < (FIELD == 1 ? 2 : 3); ++k) v[k] = fx_mul<CONJ>(v[k], su3d_b<FIELD>(a, x, k), bad);
}
// v_k <- v_k conj(b_r)
template <int FIELD>
__device__ __forceinline__ void su3d_scale_row(const Ctx& a, int x, int r, FxC v[3], uint32_t& bad) {
  if (FIELD == 1 && r == 2) return;
  const FxC b = su3d_b<FIELD>(a, x, r);
#pragma unroll
  for (int k = 0; k < 3; ++k) v[k] = fx_mul<true>(v[k], b, bad);
}

// Fixed-point numbers of 32 links in shared memory.
struct FxTile {
  int4 e[32];
  __device__ __forceinline__ void put(int lane, const FxC& v) { e[lane] = make_int4(v.re.hi, v.re.lo, v.im.hi, v.im.lo); }
  __device__ __forceinline__ FxC get(int lane) const {
    const int4 v = e[lane];
    return {{v.x, v.y}, {v.z, v.w}};
  }
  __device__ __forceinline__ void put64(int lane, const int64_t v[2]) {
    e[lane] = make_int4(int(v[0]), int(v[0] >> 32), int(v[1]), int(v[1] >> 32));
  }
  __device__ __forceinline__ void add64(int lane, int64_t v[2]) const {
    const int4 w = e[lane];
    v[0] += (int64_t(w.y) << 32) | uint32_t(w.x);
    v[1] += (int64_t(w.w) << 32) | uint32_t(w.z);
  }
};

// Resident CTAs per SM of three warps (80 registers; 6 with 96: overrelaxation at
// 48^3x16 1.09 against 0.99 ms).
constexpr int SU3D_CTAS = 7;

// SPLIT groups of three warps share a CTA's links, each taking every SPLIT-th
// staple; the integer sums are exact, so the result does not depend on SPLIT.
template <int SPLIT>
struct Su3dShared {
  FxTile y[SPLIT][3][3], z[SPLIT][3][3];  // then: rows of A / 8 and of U
  FxTile w[2][2];                         // a subgroup's block of U A
  int2 r[4][32];                          // its rotation
  int keep[32];                           // no rotation
  uint32_t flag[3 * SPLIT][32];
  int offset[4][2][32];                   // of the neighbour's index, forward and backward
  int64_t first[3][5][32];                // a heat-bath's draws ahead of the staples, by subgroup
};
// The plane-summing phases keep the part of the staple sum over nu < mu.
template <int SPLIT>
struct Su3dMeasShared : Su3dShared<SPLIT> {
  FxTile low[SPLIT][3][3];
  double sum[3];
};

// The rotation of subgroup `sub` from its block in sh.w into sh.r; whether all tries
// of a heat-bath failed (FX_EXHAUSTED), or the block or the draw is too small for fixed
// point (FX_SMALL_DRAW: the FP64 path does the update).  Out of line: one copy for the
// three subgroups.
template <int KIND, int SPLIT>
__device__ __noinline__ unsigned su3d_rotation(Su3dShared<SPLIT>& sh, int lane, int sub, double beta, int nhit,
                                               uint32_t k0, uint32_t k1, uint32_t site, uint32_t sweep, int mu) {
  const FxC wii = sh.w[0][0].get(lane), wji = sh.w[0][1].get(lane), wij = sh.w[1][0].get(lane),
            wjj = sh.w[1][1].get(lane);
  // twice the block's quaternion over 8: k = 4 |w|
  int64_t w[4] = {fx_value(wii.re) + fx_value(wjj.re), fx_value(wij.im) + fx_value(wji.im),
                  fx_value(wij.re) - fx_value(wji.re), fx_value(wii.im) - fx_value(wjj.im)};
  Fx r[4] = {};
  bool keep = false;
  unsigned status = fx_small_block(w) ? FX_SMALL_DRAW : 0;
  if (KIND == KIND_HB) {
    const Stream dir = make_stream(k0, k1, site, sweep, mu, sub, KIND_DIR);
    if (beta == 0.0 || (w[0] | w[1] | w[2] | w[3]) == 0) {
      const Quat<double> R = su2_haar<double>(dir, 0u);
      uint32_t e = 0;
      r[0] = fx_load(R.q0, e);
      r[1] = fx_load(R.q1, e);
      r[2] = fx_load(R.q2, e);
      r[3] = fx_load(R.q3, e);
    } else {
      FxKpFirst f;
      f.e = __longlong_as_double(sh.first[sub][0][lane]);
      f.a3 = sh.first[sub][1][lane];
#pragma unroll
      for (int k = 0; k < 3; ++k) f.d[k] = sh.first[sub][2 + k][lane];
      // alpha = (2/3) beta k
      status |= fx_heatbath(w, 0.375 / beta, nhit, make_stream(k0, k1, site, sweep, mu, sub, KIND_TRY), f, r);
      keep = status & FX_EXHAUSTED;
    }
  } else {
    keep = !fx_overrelax(w, r);
  }
#pragma unroll
  for (int k = 0; k < 4; ++k) sh.r[k][lane] = make_int2(r[k].hi, r[k].lo);
  sh.keep[lane] = keep;
  return status;
}

__device__ __forceinline__ void bar_96(int id) { asm volatile("bar.sync %0, 96;" ::"r"(id) : "memory"); }

template <int FIELD, int KIND, int SPLIT, int INT>
__global__ void __launch_bounds__(96 * SPLIT, SU3D_CTAS / SPLIT)
    su3d_phase_kernel(const __grid_constant__ Ctx a, int parity, int mu) {
  extern __shared__ __align__(16) unsigned char smem[];
  constexpr bool meas = KIND == KIND_OR_MEAS, reunit = KIND == KIND_OR_REUNIT || meas;
  using Shared = std::conditional_t<meas, Su3dMeasShared<SPLIT>, Su3dShared<SPLIT>>;
  Shared& sh = *reinterpret_cast<Shared*>(smem);
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, group = SPLIT == 1 ? 0 : warp / 3;
  const int role = warp - 3 * group;
  const int h0 = blockIdx.x * 32 + lane, h = min(h0, a.g.Vh - 1);
  const Site x = site_of(a.g, parity, h);
  const bool on = h0 < a.g.Vh && !frozen_link(a, mu, x.t);
  if (a.field_mode == 1 && !__syncthreads_or(on)) return;
  uint32_t big = 0, bad = 0;
  const int s0 = lex(a.g, x);
  if (group == 0) {
    // index offsets to the neighbours, for two warps to look up by direction
#pragma unroll
    for (int d = 0; d < 4; ++d)
      if (role == (d & 1)) {
        const int c = d == 0 ? x.x : d == 1 ? x.y : d == 2 ? x.z : x.t;
        const int ext = d == 3 ? a.g.Nt : a.g.Ns;
        const int st = d == 0 ? 1 : d == 1 ? a.g.Ns : d == 2 ? a.g.Ns * a.g.Ns : a.g.Ns * a.g.Ns * a.g.Ns;
        sh.offset[d][0][lane] = c == ext - 1 ? st - ext * st : st;
        sh.offset[d][1][lane] = c == 0 ? ext * st - st : -st;
      }
  }
  uint32_t sweep = 0;
  if (KIND == KIND_HB) {
    sweep = *a.sweep;
    if (group == 0) {
      const FxKpFirst f = fx_kp_first(make_stream(a.k0, a.k1, uint32_t(s0), sweep, mu, role, KIND_TRY),
                                      make_stream(a.k0, a.k1, uint32_t(s0), sweep, mu, role, KIND_DIR));
      sh.first[role][0][lane] = __double_as_longlong(f.e);
      sh.first[role][1][lane] = f.a3;
#pragma unroll
      for (int k = 0; k < 3; ++k) sh.first[role][2 + k][lane] = f.d[k];
    }
  }
  __syncthreads();
  const int64_t plane = a.g.plane;
  const double2* links = reinterpret_cast<const double2*>(a.links);
  auto link = [&](int m, int p, int s) { return links + (m * 2 + p) * plane + (s >> 1); };
  const int up = sh.offset[mu][0][lane];
  // x coordinate one step along mu
  const int x_mu = mu == 0 ? (x.x == a.g.Ns - 1 ? 0 : x.x + 1) : x.x;

  int64_t A[3][2] = {};  // row `role` of the staple sum
#pragma unroll 1
  for (int s = group; s < 6; s += SPLIT) {
    // Both kinds of staple are X Y^+ Z^+: Ut_nu(x+mu) Ut_mu(x+nu)^+ Ut_nu(x)^+,
    // and (Ut_mu(x-nu) Ut_nu(x+mu-nu))^+ Ut_nu(x-nu) with X and Z the adjoints
    // of its nu-links.  The background of a y-link is a diagonal factor on its
    // right: it multiplies columns, or rows of the adjoint.
    const int n = s >> 1, nu = n + (n >= mu);
    const bool lower = s & 1;
    const int off = sh.offset[nu][s & 1][lane];
    const int base = lower ? s0 + off : s0, pb = parity ^ (s & 1);
    const RawRow wx = su3d_row(a, link(nu, pb ^ 1, base + up), role, lower);
    const RawRow wy = su3d_row(a, link(mu, parity ^ 1, s0 + off), role, false);
    const RawRow wz = su3d_row(a, link(nu, pb, base), role, lower);
    FxC X[3], V[3];
    su3d_convert<(INT & 1)>(wx, lower, X, big);
    su3d_convert<(INT >> 1 & 1)>(wy, false, V, big);
    if (s >= SPLIT) bar_96(1 + group);  // the tiles' readers are done
#pragma unroll
    for (int k = 0; k < 3; ++k) sh.y[group][role][k].put(lane, V[k]);
    su3d_convert<(INT >> 2 & 1)>(wz, lower, V, big);
    if (FIELD && nu == 1 && lower) su3d_scale_row<FIELD>(a, x.x, role, V, bad);
#pragma unroll
    for (int k = 0; k < 3; ++k) sh.z[group][role][k].put(lane, V[k]);
    if (FIELD && mu == 1) {
      const int xn = nu > 0 ? x.x : lower ? (x.x == 0 ? a.g.Ns - 1 : x.x - 1) : (x.x == a.g.Ns - 1 ? 0 : x.x + 1);
      su3d_scale<FIELD, true>(a, xn, X, bad);
    }
    if (FIELD && nu == 1) {
      if (lower) su3d_scale_row<FIELD>(a, x_mu, role, X, bad);
      else su3d_scale<FIELD, false>(a, x_mu, X, bad);
    }
    bar_96(1 + group);
#pragma unroll
    for (int j = 0; j < 3; ++j) {
      FxDot<true> d;
#pragma unroll
      for (int k = 0; k < 3; ++k) d.add(X[k], sh.y[group][j][k].get(lane));
      V[j] = d.limbs(bad);
    }
    if (FIELD && nu == 1 && !lower) su3d_scale<FIELD, true>(a, x.x, V, bad);
#pragma unroll
    for (int j = 0; j < 3; ++j) {
      FxDot<true> d;
#pragma unroll
      for (int k = 0; k < 3; ++k) d.add(V[k], sh.z[group][j][k].get(lane));
      const int64_t re = d.re(), im = d.im();
      fx_check(re, bad);
      fx_check(im, bad);
      A[j][0] += re;
      A[j][1] += im;
    }
    if constexpr (meas)
      if (nu < mu) {  // the last one leaves the sum so far
#pragma unroll
        for (int j = 0; j < 3; ++j) sh.low[group][role][j].put64(lane, A[j]);
      }
  }
  if constexpr (meas)
    if (group >= 2 * mu) {  // no staple with nu < mu here
      const int64_t zero[2] = {0, 0};
#pragma unroll
      for (int j = 0; j < 3; ++j) sh.low[group][role][j].put64(lane, zero);
    }
  if (SPLIT > 1) {
    bar_96(1 + group);
    if (group > 0) {
#pragma unroll
      for (int j = 0; j < 3; ++j) sh.y[group][role][j].put64(lane, A[j]);
      sh.flag[warp][lane] = (bad & FX_BAD) | (big & FX_BIG);
    }
    __syncthreads();
    if (group > 0) return;
#pragma unroll 1
    for (int g = 1; g < SPLIT; ++g) {
#pragma unroll
      for (int j = 0; j < 3; ++j) sh.y[g][role][j].add64(lane, A[j]);
      const uint32_t f = sh.flag[3 * g + role][lane];
      bad |= f & FX_BAD;
      big |= f & FX_BIG;
    }
  }

  // Rows to shared memory: B A / 8 (Ut A = U (B A); below 2 in magnitude) and U.
  FxC U[3], W[3];
  {
    su3d_convert<(INT & 1)>(su3d_row(a, link(mu, parity, s0), role, false), false, U, big);
#pragma unroll
    for (int j = 0; j < 3; ++j) W[j] = {fx_limbs(A[j][0] >> 3), fx_limbs(A[j][1] >> 3)};
    if (FIELD && mu == 1 && (FIELD == 2 || role < 2)) {
      const FxC b = su3d_b<FIELD>(a, x.x, role);
#pragma unroll
      for (int j = 0; j < 3; ++j) W[j] = fx_mul<false>(W[j], b, bad);
    }
    bar_96(1);
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      sh.y[0][role][k].put(lane, W[k]);
      sh.z[0][role][k].put(lane, U[k]);
    }
    bar_96(1);
    // column `role` of Ut A / 8 and of U
    FxC F[3];
#pragma unroll
    for (int k = 0; k < 3; ++k) F[k] = sh.y[0][k][role].get(lane);
#pragma unroll
    for (int i = 0; i < 3; ++i) {
      FxDot<false> d;
#pragma unroll
      for (int k = 0; k < 3; ++k) d.add(sh.z[0][i][k].get(lane), F[k]);
      W[i] = d.limbs(bad);
      U[i] = sh.z[0][i][role].get(lane);
    }
  }
  unsigned status = 0;
#pragma unroll
  for (int sub = 0; sub < 3; ++sub) {
    const int i = sub == 1 ? 1 : 0;
    const int j = sub == 0 ? 1 : 2;
    if (role == i || role == j) {
      sh.w[role == j][0].put(lane, W[i]);
      sh.w[role == j][1].put(lane, W[j]);
    }
    bar_96(1);
    if (role == sub)
      status = su3d_rotation<KIND, SPLIT>(sh, lane, sub, a.beta, a.nhit, a.k0, a.k1, uint32_t(s0), sweep, mu);
    bar_96(1);
    if (!sh.keep[lane]) {
      Fx r[4];
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        const int2 v = sh.r[k][lane];
        r[k] = {v.x, v.y};
      }
      const FxC r00{r[0], r[3]}, r01{r[2], r[1]}, r10{fx_neg(r[2]), r[1]}, r11{r[0], fx_neg(r[3])};
      auto rotate = [&](FxC v[3]) {
        FxDot<false> di, dj;
        di.add(r00, v[i]);
        di.add(r01, v[j]);
        dj.add(r10, v[i]);
        dj.add(r11, v[j]);
        v[i] = di.limbs(bad);
        v[j] = dj.limbs(bad);
      };
      rotate(U);
      if (sub < 2) rotate(W);
    }
  }

  if (status & FX_SMALL_DRAW) bad |= FX_BAD;
  sh.flag[role][lane] = (bad & FX_BAD) | (big & FX_BIG);
  if (reunit) {
#pragma unroll
    for (int i = 0; i < 3; ++i) sh.y[0][i][role].put(lane, U[i]);
  }
  bar_96(1);
  const bool out_of_range = sh.flag[0][lane] | sh.flag[1][lane] | sh.flag[2][lane];
  if (!meas && !on) return;
  double v64 = 0.0;  // Re Tr of an FP64 update
  if (on && out_of_range) {
    if (role == 0) v64 = su3_update_fp64<double, FIELD, KIND>(a, parity, mu, h);
  } else if (on) {
    if (status & FX_EXHAUSTED) atomicAdd(a.exhausted, 1ull);
    if (!reunit) {
      double2* out = reinterpret_cast<double2*>(a.links);
#pragma unroll
      for (int i = 0; i < 3; ++i)
        out[vidx(a.g, 3 * i + role, mu, parity, h)] =
            make_double2(fx_double(fx_value(U[i].re)), fx_double(fx_value(U[i].im)));
    } else if (role == 0) {
      FxC m[3][3];
#pragma unroll
      for (int i = 0; i < 3; ++i)
#pragma unroll
        for (int k = 0; k < 3; ++k) m[i][k] = sh.y[0][i][k].get(lane);
      M3<double> d;
      auto to_double = [&]() {
#pragma unroll
        for (int i = 0; i < 3; ++i)
#pragma unroll
          for (int k = 0; k < 3; ++k) d.e[i][k] = {fx_double(fx_value(m[i][k].re)), fx_double(fx_value(m[i][k].im))};
      };
      if (fx_reunit(m)) {
        to_double();
      } else {  // rows far from unitary
#pragma unroll
        for (int i = 0; i < 3; ++i)
#pragma unroll
          for (int k = 0; k < 3; ++k) m[i][k] = sh.y[0][i][k].get(lane);
        to_double();
        su3d_reunit(d);
        if (meas)
#pragma unroll
          for (int i = 0; i < 3; ++i)
#pragma unroll
            for (int k = 0; k < 3; ++k) m[i][k] = {fx_load(d.e[i][k].re, big), fx_load(d.e[i][k].im, big)};
      }
      SU3Policy<double>::store(a.links, a.g, mu, parity, h, d);
      if (meas)
#pragma unroll
        for (int i = 0; i < 3; ++i)
#pragma unroll
          for (int k = 0; k < 3; ++k) sh.z[0][i][k].put(lane, m[i][k]);
    }
  }
  if constexpr (meas) {
    bar_96(1);
    // column `role` of the final effective link times row `role` of the partial sum
    FxAcc p, q;
    if (on && !out_of_range) {
      FxC u[3];
#pragma unroll
      for (int i = 0; i < 3; ++i) u[i] = sh.z[0][i][role].get(lane);
      if (FIELD && mu == 1 && (FIELD == 2 || role < 2)) {
        const FxC b = su3d_b<FIELD>(a, x.x, role);
#pragma unroll
        for (int i = 0; i < 3; ++i) u[i] = fx_mul<false>(u[i], b, bad);
      }
#pragma unroll
      for (int i = 0; i < 3; ++i) {
        int64_t t[2] = {0, 0};
        for (int g = 0; g < SPLIT; ++g) sh.low[g][role][i].add64(lane, t);
        p.add(u[i].re, fx_limbs(t[0] >> 3));
        q.add(u[i].im, fx_limbs(t[1] >> 3));
      }
    }
    double s = 8.0 * fx_warp_sum(fx_diff(p, q));
    if (role == 0 && __any_sync(0xffffffffu, on && out_of_range)) {
#pragma unroll
      for (int off = 16; off > 0; off >>= 1) v64 += __shfl_down_sync(0xffffffffu, v64, off);
      s += v64;
    }
    if (lane == 0) sh.sum[role] = s;
    bar_96(1);
    if (threadIdx.x == 0) a.partials[fused_plaq_offset(a.g, mu) + blockIdx.x] = sh.sum[0] + sh.sum[1] + sh.sum[2];
  }
}

// Three warps with 32 sites; the sums of Re and Im Tr over the warp's lanes.
struct Su3dMeasTiles {
  FxTile t[2][3][3];
  uint32_t flag[3][32];
};

// FP64 for sites out of the fixed-point range, out of line.
static __device__ __noinline__ double2 su3d_poly_fp64(const Ctx& a, int site) {
  SumD v0, v1;
  polyakov_site<SU3Policy<double>>(a, site, v0, v1);
  return make_double2(v0.s, v1.s);
}

// Polyakov loop of 32 spatial sites: warp r with row r of the running product over
// t; each converts row r of the next link for the three.
__device__ __forceinline__ void su3d_poly(const Ctx& a, int base, Su3dMeasTiles& sh, int role, int lane, int bar,
                                          double& re, double& im) {
  const int Ns = a.g.Ns, V3 = Ns * Ns * Ns;
  const int site = base + lane, s0 = min(site, V3 - 1);
  const int xyz = s0 % Ns + s0 / Ns % Ns + s0 / (Ns * Ns);
  const double2* links = reinterpret_cast<const double2*>(a.links) + 6 * a.g.plane;
  auto row = [&](int t) {
    const int64_t s = s0 + int64_t(t) * V3;
    return su3d_row(a, links + ((xyz + t) & 1) * a.g.plane + (s >> 1), role, false);
  };
  uint32_t big = 0, bad = 0;
  FxC v[3], w[3];
  su3d_convert<1>(row(0), false, v, big);
  RawRow next = row(1);
#pragma unroll 1
  for (int t = 1; t < a.g.Nt; ++t) {
    su3d_convert<1>(next, false, w, big);
    if (t + 1 < a.g.Nt) next = row(t + 1);
#pragma unroll
    for (int k = 0; k < 3; ++k) sh.t[t & 1][role][k].put(lane, w[k]);
    bar_96(bar);  // (the other buffer's readers passed this one's predecessor)
#pragma unroll
    for (int j = 0; j < 3; ++j) {
      FxDot<false> d;
#pragma unroll
      for (int k = 0; k < 3; ++k) d.add(v[k], sh.t[t & 1][k][j].get(lane));
      w[j] = d.limbs(bad);
    }
#pragma unroll
    for (int k = 0; k < 3; ++k) v[k] = w[k];
  }
  uint32_t parts = 0;
#pragma unroll
  for (int k = 0; k < 3; ++k) parts |= fx_part(v[k].re) | fx_part(v[k].im);
  if (fx_tiny(parts)) bad |= FX_BAD;
  sh.flag[role][lane] = (bad & FX_BAD) | (big & FX_BIG);
  bar_96(bar);
  const bool in = site < V3, out_of_range = sh.flag[0][lane] | sh.flag[1][lane] | sh.flag[2][lane];
  const FxC d = role == 0 ? v[0] : role == 1 ? v[1] : v[2];
  const bool fixed = in && !out_of_range;
  re = fx_warp_sum(fixed ? fx_value(d.re) : 0);
  im = fx_warp_sum(fixed ? fx_value(d.im) : 0);
  if (role == 0 && __any_sync(0xffffffffu, in && out_of_range)) {
    SumD v0, v1;
    if (in && out_of_range) {
      const double2 v = su3d_poly_fp64(a, site);
      v0.s = v.x;
      v1.s = v.y;
    }
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) {
      v0.merge_down(off);
      v1.merge_down(off);
    }
    re += v0.s;
    im += v1.s;
  }
}

// Polyakov loop of a working sweep's fused measurement, 32 spatial sites per CTA.
// FP64 block partials of Tr, in a fixed order.  (The plane sums, this kernel and the
// final sums add 41 us to a sweep of 16^3x4 and 77 to one of 32^3x8; the separate
// FP64 measurement took 128 and 780.)
static __global__ void __launch_bounds__(96) su3d_poly_kernel(const __grid_constant__ Ctx a) {
  __shared__ Su3dMeasTiles sh;
  __shared__ double sum[3][2];
  const int lane = threadIdx.x & 31, role = threadIdx.x >> 5;
  double re, im;
  su3d_poly(a, blockIdx.x * 32, sh, role, lane, 1, re, im);
  if (lane == 0) {
    sum[role][0] = re;
    sum[role][1] = im;
  }
  __syncthreads();
  if (threadIdx.x < 2)
    a.partials[fused_plaq_offset(a.g, 4) + 2 * blockIdx.x + threadIdx.x] =
        sum[0][threadIdx.x] + sum[1][threadIdx.x] + sum[2][threadIdx.x];
}

inline cudaError_t su3d_measure_fused_tail(const Ctx& a, int /*block*/, cudaStream_t st) {
  const int nl = fused_poly32_blocks(a.g);
  su3d_poly_kernel<<<nl, 96, 0, st>>>(a);
  launch_fused_final(a, st, (a.g.Vh + 31) / 32, 3.0, nl, fused_plaq_offset(a.g, 4), 3.0);
  return cudaGetLastError();
}

template <int FIELD, int KIND, int SPLIT, int INT>
inline cudaError_t su3d_launch_one(const Ctx& a, int parity, int mu, cudaStream_t st) {
  constexpr int bytes = int(KIND == KIND_OR_MEAS ? sizeof(Su3dMeasShared<SPLIT>) : sizeof(Su3dShared<SPLIT>));
  if (bytes > 48 * 1024) {
    const cudaError_t e = cudaFuncSetAttribute(su3d_phase_kernel<FIELD, KIND, SPLIT, INT>,
                                               cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
    if (e != cudaSuccess) return e;
  }
  su3d_phase_kernel<FIELD, KIND, SPLIT, INT><<<(a.g.Vh + 31) / 32, 96 * SPLIT, bytes, st>>>(a, parity, mu);
  return cudaGetLastError();
}

// The split that leaves every CTA resident in one wave of the 152 SMs: 6 up to
// one CTA (of 18 warps) per SM, 2 up to three (of 6 warps) per SM.  Sweeps of
// 1 heat-bath + 4 overrelaxation passes, us, split 6 / 2 / 1 at 4^3x4: 436 / 508 /
// 678; 12^3x4 (108 CTAs): 456 / 534 / 726; 14^3x4 (172): 842 / 679 / 858; 16^3x6
// (384): 1254 / 933 / 1072; 20^3x4 (500): 1648 / 1312 / 1120; 32^3x8: 11847 / 7394 /
// 6400.  (A split of 3 was never the best by more than 2 %.)
//
// Conversions: on the integer pipe for the split kernels (few warps: one on the
// FP64 unit holds its warp for 64 cycles); at full occupancy Z's go to the FP64
// unit, which is otherwise idle (32^3x8 overrelaxation 151 -> 146 us; X's or Y's
// too: 149).
template <int FIELD, int KIND>
inline cudaError_t su3d_launch_kind(const Ctx& a, int parity, int mu, cudaStream_t st) {
  const int groups = (a.g.Vh + 31) / 32;
  if (groups <= GB300_SMS) return su3d_launch_one<FIELD, KIND, 6, 7>(a, parity, mu, st);
  if (groups <= 3 * GB300_SMS) return su3d_launch_one<FIELD, KIND, 2, 7>(a, parity, mu, st);
  return su3d_launch_one<FIELD, KIND, 1, 3>(a, parity, mu, st);
}

template <int KIND>
inline cudaError_t su3d_launch_level(const Ctx& a, int parity, int mu, cudaStream_t st) {
  switch (su3_field_level(a)) {
    case 0: return su3d_launch_kind<0, KIND>(a, parity, mu, st);
    case 1: return su3d_launch_kind<1, KIND>(a, parity, mu, st);
    default: return su3d_launch_kind<2, KIND>(a, parity, mu, st);
  }
}

// Heat-bath, the reunitarizing overrelaxation and what measures are compiled in
// translation units of their own.
cudaError_t su3d_launch_hb(const Ctx& a, int parity, int mu, cudaStream_t st);
cudaError_t su3d_launch_or_reunit(const Ctx& a, int parity, int mu, cudaStream_t st);
cudaError_t su3d_launch_or_meas(const Ctx& a, int parity, int mu, cudaStream_t st);
cudaError_t su3d_launch_measure(const Ctx& a, int effective, cudaStream_t st);

}  // namespace qcd
