// qcd_su2d.cuh -- SU(2) phase update with FP64 links, its quaternion products in
// fixed point (qcd_fix.cuh) on the integer pipe; the counterpart of qcd_su2c.cuh
// for the single-lattice kernels and the batched kernel (CG: loads through L2).
#pragma once

#include "qcd_fixmath.cuh"
#include "qcd_su2c.cuh"

namespace qcd {

// Quaternion of a link, conjugated with DAG.  Conversions on the integer pipe:
// a third of them on the FP64 unit was no faster at 64^3x16 and 14 % slower at
// 20^3x4, two thirds slower everywhere.
template <bool DAG, bool CG>
__device__ __forceinline__ void su2d_load(const Ctx& a, int d, int par, int s, Fx q[4], uint32_t& big) {
  const Quat<double> u = SU2Policy<double>::template load<CG>(a.links, a.g, d, par, s >> 1);
  const double v[4] = {u.q0, DAG ? -u.q1 : u.q1, DAG ? -u.q2 : u.q2, DAG ? -u.q3 : u.q3};
#pragma unroll
  for (int k = 0; k < 4; ++k) q[k] = fx_load_int(v[k], big);
}

// q (c + s k), or with LEFT (c - s k) q, the adjoint of q^+ (c + s k); with
// INVERSE the sign of s turned.
template <bool LEFT, bool INVERSE>
__device__ __forceinline__ void su2d_phase(const Ctx& a, int x, Fx q[4], uint32_t& bad) {
  uint32_t e = 0;
  const double2 v = __ldg(a.phase64 + x);
  const Fx c = fx_load_int(v.x, e), s = fx_load_int(LEFT != INVERSE ? -v.y : v.y, e), n = fx_neg(s);
  FxAcc r[4];
#pragma unroll
  for (int k = 0; k < 4; ++k) r[k].add(q[k], c);
  r[0].add(q[3], n);
  r[3].add(q[0], s);
  r[1].add(q[2], LEFT ? s : n);
  r[2].add(q[1], LEFT ? n : s);
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    const int64_t t = r[k].value();
    fx_check(t, bad);
    q[k] = fx_limbs(t);
  }
}

template <bool FIELD, int D, bool DAG, bool CG>
__device__ __forceinline__ void su2d_eff(const Ctx& a, int par, const LexSite& x, Fx q[4], uint32_t& big,
                                         uint32_t& bad) {
  su2d_load<DAG, CG>(a, D, par, x.s, q, big);
  if (FIELD && D == 1) su2d_phase<DAG, false>(a, x.c[0], q, bad);
}

// A += one staple of U_MU(x): Ut_nu(x+mu) Ut_mu(x+nu)^+ Ut_nu(x)^+, or
// Ut_nu(x+mu-nu)^+ Ut_mu(x-nu)^+ Ut_nu(x-nu).
template <bool FIELD, int MU, int NU, bool LOWER, bool CG>
__device__ __forceinline__ void su2d_staple(const Ctx& a, int p, const LexSite& x, int64_t A[4], uint32_t& big,
                                            uint32_t& bad) {
  const LexSite xn = lex_step<NU, LOWER ? -1 : +1>(a.g, x);
  const LexSite& base = LOWER ? xn : x;
  const LexSite xp = lex_step<MU, +1>(a.g, base);
  const int pb = LOWER ? p ^ 1 : p;
  Fx u[4], v[4];
  int64_t t[4];
  su2d_eff<FIELD, NU, LOWER, CG>(a, pb ^ 1, xp, u, big, bad);
  su2d_eff<FIELD, MU, true, CG>(a, p ^ 1, xn, v, big, bad);
  fx_qmul(u, v, t);
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    fx_check(t[k], bad);
    u[k] = fx_limbs(t[k]);
  }
  su2d_eff<FIELD, NU, !LOWER, CG>(a, pb, base, v, big, bad);
  fx_qmul(u, v, t);
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    fx_check(t[k], bad);
    A[k] += t[k];
  }
}

// The update in FP64, out of line: links outside the fixed-point range.
template <bool FIELD, int KIND, bool CG>
__device__ __noinline__ double su2d_general(Ctx a, int parity, int mu, LexSite x, uint32_t sweep) {
  switch (mu) {
    case 0: return su2c_update_at<double, FIELD, KIND, 0, CG>(a, parity, x, sweep);
    case 1: return su2c_update_at<double, FIELD, KIND, 1, CG>(a, parity, x, sweep);
    case 2: return su2c_update_at<double, FIELD, KIND, 2, CG>(a, parity, x, sweep);
    default: return su2c_update_at<double, FIELD, KIND, 3, CG>(a, parity, x, sweep);
  }
}

static __device__ __noinline__ Quat<double> su2d_haar(Stream dir) { return su2_haar<double>(dir, 0u); }

// One link update given its staple sum A (and the part of it over nu < MU), as
// su2c_update_at.
template <bool FIELD, int KIND, bool CG>
__device__ __forceinline__ double su2d_update(const Ctx& a, int parity, int mu, const LexSite& x, uint32_t sweep,
                                              int64_t A[4], const int64_t low[4], uint32_t big, uint32_t bad,
                                              const FxKpFirst* first) {
  constexpr bool reunit = KIND == KIND_OR_REUNIT || KIND == KIND_OR_MEAS;
  constexpr bool meas = KIND == KIND_OR_MEAS;
  const bool phased = FIELD && mu == 1;
  using P = SU2Policy<double>;
  Fx u[4];
  bool general = (bad & FX_BAD) || (big & FX_BIG) || fx_small(A);
  if (KIND == KIND_HB) {
    const Stream dir = make_stream(a.k0, a.k1, uint32_t(x.s), sweep, mu, 0, KIND_DIR);
    if (a.beta == 0.0) {
      const Quat<double> R = su2d_haar(dir);
      u[0] = fx_load(R.q0, big);
      u[1] = fx_load(R.q1, big);
      u[2] = fx_load(R.q2, big);
      u[3] = fx_load(R.q3, big);
      general = false;
    } else if (!general) {
      const Stream tries = make_stream(a.k0, a.k1, uint32_t(x.s), sweep, mu, 0, KIND_TRY);
      const int status = fx_heatbath(A, 1.0 / a.beta, a.nhit, tries, *first, u);
      if (status == FX_EXHAUSTED) {
        atomicAdd(a.exhausted, 1ull);
        return 0.0;  // the link stays as it is
      }
      general = status == FX_SMALL_DRAW;
    }
    if (general) return su2d_general<FIELD, KIND, CG>(a, parity, mu, x, sweep);
  } else {
    if (general) return su2d_general<FIELD, KIND, CG>(a, parity, mu, x, sweep);
    su2d_load<false, CG>(a, mu, parity, x.s, u, big);
    const bool tiny = fx_tiny(fx_part(u[0]) | fx_part(u[1]) | fx_part(u[2]) | fx_part(u[3]));
    if (phased) su2d_phase<false, false>(a, x.c[0], u, bad);
    fx_reflect(A, u, bad);
    if (tiny || (bad & FX_BAD) || (big & FX_BIG)) return su2d_general<FIELD, KIND, CG>(a, parity, mu, x, sweep);
  }
  // Ut_new B^+ (components below 2 before, so below 4 = 2^60 and within two limbs after)
  if (phased) su2d_phase<false, true>(a, x.c[0], u, bad);
  Quat<double> q;
  bool done = false;
  if (reunit) {
    FxAcc n;
#pragma unroll
    for (int k = 0; k < 4; ++k) n.add(u[k], u[k]);
    Fx d;
    done = fx_unit_factor(n.value(), d);
    if (done)
#pragma unroll
      for (int k = 0; k < 4; ++k) u[k] = fx_scale1p(u[k], d);
  }
  q = {fx_double(fx_value(u[0])), fx_double(fx_value(u[1])), fx_double(fx_value(u[2])), fx_double(fx_value(u[3]))};
  if (reunit && !done) {
    q = su2_reunit_value<double>(q);
    u[0] = fx_load(q.q0, big);
    u[1] = fx_load(q.q1, big);
    u[2] = fx_load(q.q2, big);
    u[3] = fx_load(q.q3, big);
  }
  P::store(a.links, a.g, mu, parity, x.s >> 1, q);
  if (!meas) return 0.0;
  if (phased) su2d_phase<false, false>(a, x.c[0], u, bad);
  FxAcc t;  // (1/2) Re Tr(Ut low) / 8
#pragma unroll
  for (int k = 0; k < 4; ++k) t.add(u[k], fx_limbs(k ? -(low[k] >> 3) : low[k] >> 3));
  return 8.0 * fx_double(t.value());
}

// The whole update by one thread.
template <bool FIELD, int KIND, int MU, bool CG>
__device__ __forceinline__ double su2d_update_at(const Ctx& a, int parity, const LexSite& x, uint32_t sweep) {
  if (frozen_link(a, MU, x.c[3])) return 0.0;
  int64_t A[4] = {}, low[4] = {};
  uint32_t big = 0, bad = 0;
#pragma unroll
  for (int n = 0; n < 3; ++n) {
    if (n == MU)
#pragma unroll
      for (int k = 0; k < 4; ++k) low[k] = A[k];
    switch (n + (n >= MU)) {
#define QCD_SU2D_NU(NU)                                                                \
  case NU:                                                                             \
    if (NU != MU) {                                                                    \
      su2d_staple<FIELD, MU, NU, false, CG>(a, parity, x, A, big, bad);          \
      su2d_staple<FIELD, MU, NU, true, CG>(a, parity, x, A, big, bad);           \
    }                                                                                  \
    break;
      QCD_SU2D_NU(0)
      QCD_SU2D_NU(1)
      QCD_SU2D_NU(2)
      QCD_SU2D_NU(3)
#undef QCD_SU2D_NU
    }
  }
  if (MU == 3)
#pragma unroll
    for (int k = 0; k < 4; ++k) low[k] = A[k];
  FxKpFirst first;
  if (KIND == KIND_HB)
    first = fx_kp_first(make_stream(a.k0, a.k1, uint32_t(x.s), sweep, MU, 0, KIND_TRY),
                        make_stream(a.k0, a.k1, uint32_t(x.s), sweep, MU, 0, KIND_DIR));
  return su2d_update<FIELD, KIND, CG>(a, parity, MU, x, sweep, A, low, big, bad, &first);
}

// Bound: integer pipe and FP64 unit together (ncu at 32^3x8, overrelaxation of
// t-links: ALU 45 %, 3,390 instructions per update) where the FP64 form was bound
// by the FP64 unit.  Phase times, us, FP64 form -> this, overrelaxation /
// heat-bath of y-links: 32^3x8 77 / 159 -> 32 / 42;
// 64^3x16 1104 / 2135 -> 406 / 529.  128 registers: with 96 / 80 / 64 sweeps took
// 1.00 / 1.04 / 1.15 times as long at 64^3x16 and 1.07 / 1.20 / 1.15 at 32^3x8.
//
// One thread per link.
template <bool FIELD, int KIND, int MU>
__global__ void __maxnreg__(128) su2d_phase_kernel(const __grid_constant__ Ctx a, int parity) {
  SumD v[1];
  const int h = blockIdx.x * blockDim.x + threadIdx.x;
  if (h < a.g.Vh)
    v[0].s = su2d_update_at<FIELD, KIND, MU, false>(a, parity, lex_site(a, parity, h), KIND == KIND_HB ? *a.sweep : 0u);
  if (KIND == KIND_OR_MEAS) block_sums(v, a.partials + fused_plaq_offset(a.g, MU) + blockIdx.x);
}

// Small lattices: six warps share 32 links, each taking one staple; the integer
// sums are exact, so the results are the same.  The directions are run-time values
// and the two kinds of staple one body (the adjoint of a link by the sign of its
// imaginary quaternion parts), so that the code stays in the instruction caches
// from phase to phase (a kernel per direction with a body per staple took 1.1 / 1.4 /
// 1.5 times as long per sweep at 4^3x4 / 12^3x4 / 16^3x4).
__device__ __forceinline__ void su2d_load_at(const Ctx& a, int d, int par, int s, uint32_t dag, Fx q[4], uint32_t& big) {
  const Quat<double> u = SU2Policy<double>::load(a.links, a.g, d, par, s >> 1);
  const double v[4] = {u.q0, u.q1, u.q2, u.q3};
#pragma unroll
  for (int k = 0; k < 4; ++k)
    q[k] = fx_load_int(k ? __hiloint2double(__double2hiint(v[k]) ^ int(dag), __double2loint(v[k])) : v[k], big);
}

template <bool FIELD, int KIND>
__global__ void __launch_bounds__(192) su2d_split_kernel(const __grid_constant__ Ctx a, int parity, int mu) {
  __shared__ int64_t part[6][4][32];
  __shared__ uint32_t flag[6][32];
  __shared__ FxKpFirst ahead[32];
  const int lane = threadIdx.x & 31, role = threadIdx.x >> 5;
  const int h = blockIdx.x * 32 + lane;
  const bool in = h < a.g.Vh;
  const LexSite x = lex_site(a, parity, in ? h : a.g.Vh - 1);
  const bool on = in && !frozen_link(a, mu, x.c[3]);
  const uint32_t sweep = KIND == KIND_HB ? *a.sweep : 0u;
  int64_t A[4] = {};
  uint32_t big = 0, bad = 0;
  {
    const int n = role >> 1, nu = n + (n >= mu);
    const bool lower = role & 1;
    auto stride = [&](int d) { return d == 0 ? 1 : d == 1 ? a.g.Ns : d == 2 ? a.g.Ns * a.g.Ns : a.g.Ns * a.g.Ns * a.g.Ns; };
    auto coord = [&](int d) { return d == 0 ? x.c[0] : d == 1 ? x.c[1] : d == 2 ? x.c[2] : x.c[3]; };
    const int st_mu = stride(mu), st_nu = stride(nu), c_mu = coord(mu), c_nu = coord(nu);
    const int e_mu = mu == 3 ? a.g.Nt : a.g.Ns, e_nu = nu == 3 ? a.g.Nt : a.g.Ns;
    const int up = c_mu == e_mu - 1 ? st_mu - e_mu * st_mu : st_mu;
    const int off =
        lower ? (c_nu == 0 ? e_nu * st_nu - st_nu : -st_nu) : (c_nu == e_nu - 1 ? st_nu - e_nu * st_nu : st_nu);
    const int base = lower ? x.s + off : x.s, pb = lower ? parity ^ 1 : parity;
    const uint32_t sign = 0x80000000u;
    // Ut_nu(x+mu) Ut_mu(x+nu)^+ Ut_nu(x)^+, Ut_nu(x+mu-nu)^+ Ut_mu(x-nu)^+ Ut_nu(x-nu)
    Fx u[4], v[4], w[4];
    su2d_load_at(a, nu, pb ^ 1, base + up, lower ? sign : 0u, u, big);
    su2d_load_at(a, mu, parity ^ 1, x.s + off, sign, v, big);
    su2d_load_at(a, nu, pb, base, lower ? 0u : sign, w, big);
    if (FIELD && nu == 1) {
      const int x_mu = x.c[0] + (mu == 0 ? up : 0);
      if (lower) {
        su2d_phase<true, false>(a, x_mu, u, bad);
        su2d_phase<false, false>(a, x.c[0], w, bad);
      } else {
        su2d_phase<false, false>(a, x_mu, u, bad);
        su2d_phase<true, false>(a, x.c[0], w, bad);
      }
    }
    if (FIELD && mu == 1) su2d_phase<true, false>(a, x.c[0] + (nu == 0 ? off : 0), v, bad);
    int64_t t[4];
    fx_qmul(u, v, t);
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      fx_check(t[k], bad);
      u[k] = fx_limbs(t[k]);
    }
    fx_qmul(u, w, A);
#pragma unroll
    for (int k = 0; k < 4; ++k) fx_check(A[k], bad);
  }
#pragma unroll
  for (int k = 0; k < 4; ++k) part[role][k][lane] = A[k];
  flag[role][lane] = (bad & FX_BAD) | (big & FX_BIG);
  if (KIND == KIND_HB && role == 5)
    ahead[lane] = fx_kp_first(make_stream(a.k0, a.k1, uint32_t(x.s), sweep, mu, 0, KIND_TRY),
                              make_stream(a.k0, a.k1, uint32_t(x.s), sweep, mu, 0, KIND_DIR));
  __syncthreads();
  if (role > 0) return;
  int64_t low[4] = {};
#pragma unroll
  for (int s = 1; s < 6; ++s) {
    if (KIND == KIND_OR_MEAS && s == 2 * mu)
#pragma unroll
      for (int k = 0; k < 4; ++k) low[k] = A[k];
#pragma unroll
    for (int k = 0; k < 4; ++k) A[k] += part[s][k][lane];
    bad |= flag[s][lane] & FX_BAD;
    big |= flag[s][lane] & FX_BIG;
  }
  if (KIND == KIND_OR_MEAS && mu == 3)
#pragma unroll
    for (int k = 0; k < 4; ++k) low[k] = A[k];
  double v = 0.0;
  if (on) v = su2d_update<FIELD, KIND, false>(a, parity, mu, x, sweep, A, low, big, bad, &ahead[lane]);
  if (KIND == KIND_OR_MEAS) {  // one warp is left
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
    if (threadIdx.x == 0) a.partials[fused_plaq_offset(a.g, mu) + blockIdx.x] = v;
  }
}

// Split up to 512 CTAs of 32 links: sweeps of 1 heat-bath + 1 overrelaxation pass,
// us, split / not: 4^3x4 71 / 130, 12^3x4 (108 CTAs) 82 / 142, 16^3x4 (256) 89 / 142,
// 20^3x4 (500) 141 / 149.
inline bool su2d_split(const GeomH& g) { return (g.Vh + 31) / 32 <= 512; }
// Links of one CTA for a block size of the caller.
inline int su2d_links_per_cta(const GeomH& g, int block) { return su2d_split(g) ? 32 : block; }

template <bool FIELD, int KIND>
inline void su2d_launch_kind(const Ctx& a, int parity, int mu, int block, cudaStream_t st) {
  const unsigned grid = grid_for(a.g.Vh, su2d_links_per_cta(a.g, block));
  if (su2d_split(a.g)) {
    su2d_split_kernel<FIELD, KIND><<<grid, 192, 0, st>>>(a, parity, mu);
    return;
  }
  switch (mu) {
    case 0:
      if constexpr (KIND != KIND_OR_MEAS) su2d_phase_kernel<FIELD, KIND, 0><<<grid, block, 0, st>>>(a, parity);
      break;
    case 1: su2d_phase_kernel<FIELD, KIND, 1><<<grid, block, 0, st>>>(a, parity); break;
    case 2: su2d_phase_kernel<FIELD, KIND, 2><<<grid, block, 0, st>>>(a, parity); break;
    default: su2d_phase_kernel<FIELD, KIND, 3><<<grid, block, 0, st>>>(a, parity); break;
  }
}

template <int KIND>
inline cudaError_t su2d_launch_level(const Ctx& a, int parity, int mu, int block, cudaStream_t st) {
  if (phases_on_links(a)) su2d_launch_kind<true, KIND>(a, parity, mu, block, st);
  else su2d_launch_kind<false, KIND>(a, parity, mu, block, st);
  return cudaGetLastError();
}

}  // namespace qcd
