// on_model.cu -- the O(N) model sweep (N-component real scalar field on the
// sites, lattice phi^4 action) by multi-hit Metropolis, and its C ABI.
//
// Action:  S = sum_x [ -2 kappa sum_mu phi_x.phi_{x+mu} + phi_x.phi_x
//                      + lambda (phi_x.phi_x - 1)^2 ].
// A checkerboard phase visits every site of one parity; a visit makes nhit
// Metropolis hits with the eight neighbours fixed: hit h proposes
// phi' = phi + delta (2u - 1) componentwise (Philox block (s, sweep, 3 << 4, h))
// and accepts iff dS <= 0 or u < exp(-dS), u = word h mod 4 of block
// (s, sweep, 4 << 4, h / 4).  The local action of a value needs only
// F = sum of the neighbours: s(phi) = -2 kappa phi.F + phi.phi
// + lambda (phi.phi - 1)^2.
//
// Storage: one 16-byte vector per site and parity (FP32: float4; FP64: two
// double2 planes), even/odd halves, components beyond N kept zero.
#include <cmath>
#include <cstdarg>
#include <cstdio>
#include <cstring>
#include <limits>
#include <new>
#include <vector>

#include "qcd.h"
#include "qcd_device.cuh"

namespace qcd {
namespace {

enum : uint32_t { KIND_ON_START = 2u, KIND_ON_PROPOSE = 3u, KIND_ON_ACCEPT = 4u };

constexpr int ON_MEAS_THREADS = 256;
constexpr int ON_MEAS_VALUES = 6;  // phi.phi, hopping term, M_0..M_3

struct OnCtx {
  void* phi;
  GeomH g;
  int N;
  int nhit;
  double kappa, lambda, delta;
  float kf;  // 2 kappa for the FP32 test; NaN: every test in FP64
  uint32_t k0, k1;
  const uint32_t* sweep;
  uint32_t* sweep_rw;
  unsigned long long* accepted;
  double* partials;
  double* meas_out;
};

template <typename R>
struct OnStore;

template <>
struct OnStore<float> {
  static __device__ __forceinline__ void load(const OnCtx& a, int par, int h, float v[4]) {
    const float4 x = __ldg(reinterpret_cast<const float4*>(a.phi) + par * a.g.plane + h);
    v[0] = x.x;
    v[1] = x.y;
    v[2] = x.z;
    v[3] = x.w;
  }
  static __device__ __forceinline__ void store(const OnCtx& a, int par, int h, const float v[4]) {
    reinterpret_cast<float4*>(a.phi)[par * a.g.plane + h] = make_float4(v[0], v[1], v[2], v[3]);
  }
};

template <>
struct OnStore<double> {
  static __device__ __forceinline__ void load(const OnCtx& a, int par, int h, double v[4]) {
    const double2* p = reinterpret_cast<const double2*>(a.phi);
    const double2 x = __ldg(p + par * a.g.plane + h);
    const double2 y = __ldg(p + (2 + par) * a.g.plane + h);
    v[0] = x.x;
    v[1] = x.y;
    v[2] = y.x;
    v[3] = y.y;
  }
  static __device__ __forceinline__ void store(const OnCtx& a, int par, int h, const double v[4]) {
    double2* p = reinterpret_cast<double2*>(a.phi);
    p[par * a.g.plane + h] = make_double2(v[0], v[1]);
    p[(2 + par) * a.g.plane + h] = make_double2(v[2], v[3]);
  }
};

// The Metropolis test's exponential: FP32 from the hardware approximation
// (relative error ~2^-21, so a decision can only differ from an exact one when
// u lies within ~1e-6 of exp(-dS)); FP64 from the library.
__device__ __forceinline__ float q_exp(float x) { return __expf(x); }
__device__ __forceinline__ double q_exp(double x) { return exp(x); }

// s(phi) = -2 kappa phi.F + phi.phi + lambda (phi.phi - 1)^2
template <typename R, int N>
__device__ __forceinline__ R local_action(const R phi[4], const R F[4], R two_kappa, R lambda) {
  R pf = R(0), pp = R(0);
#pragma unroll
  for (int c = 0; c < N; ++c) {
    pf = fma(phi[c], F[c], pf);
    pp = fma(phi[c], phi[c], pp);
  }
  const R d = pp - R(1);
  return fma(-two_kappa, pf, fma(lambda * d, d, pp));
}

template <typename R, int D>
__device__ __forceinline__ void add_neighbours(const OnCtx& a, int par, const LexSite& x, R F[4]) {
  R v[4];
  const LexSite p = lex_step<D, +1>(a.g, x), m = lex_step<D, -1>(a.g, x);
  OnStore<R>::load(a, par, p.s >> 1, v);
#pragma unroll
  for (int c = 0; c < 4; ++c) F[c] += v[c];
  OnStore<R>::load(a, par, m.s >> 1, v);
#pragma unroll
  for (int c = 0; c < 4; ++c) F[c] += v[c];
}

// The hits of one FP32 site visit, on the words of proposal blocks drawn ahead.
template <int N>
struct OnHitsF32 {
  float phi[4], F[4], two_kappa, lambda, delta, cur;
  __device__ __forceinline__ OnHitsF32(const OnCtx& a, const float p[4], const float f[4])
      : two_kappa(float(2.0 * a.kappa)), lambda(float(a.lambda)), delta(float(a.delta)) {
#pragma unroll
    for (int c = 0; c < 4; ++c) {
      phi[c] = p[c];
      F[c] = f[c];
    }
    cur = local_action<float, N>(phi, F, two_kappa, lambda);
  }
  __device__ __forceinline__ bool hit(const uint4& w, uint32_t aw) {
    const uint32_t wu[4] = {w.x, w.y, w.z, w.w};
    float trial[4] = {phi[0], phi[1], phi[2], phi[3]};
#pragma unroll
    for (int c = 0; c < N; ++c) trial[c] = fma(delta, fma(2.f, u01<float>(wu[c]), -1.f), phi[c]);
    const float next = local_action<float, N>(trial, F, two_kappa, lambda);
    const float dS = next - cur;
    if (!(dS <= 0.f || u01<float>(aw) < q_exp(-dS))) return false;
#pragma unroll
    for (int c = 0; c < N; ++c) phi[c] = trial[c];
    cur = next;
    return true;
  }
  __device__ __forceinline__ void flush() {}
};

// The Metropolis test in FP64 on phi = phi0 + delta K, trial = phi0 + delta T
// (delta in units of the steps' 2^-23), out of line: the FP32 test below leaves
// about one hit in a few thousand to it.
struct OnSite64 {
  double phi0[4], F[4];
};
struct OnSteps {
  int k[4], t[4];
};
template <int N>
__device__ __noinline__ bool on_test_fp64(OnSite64 s, OnSteps n, double two_kappa, double lambda, double step,
                                          uint32_t aw) {
  double phi[4], trial[4];
#pragma unroll
  for (int c = 0; c < N; ++c) {
    phi[c] = fma(step, double(n.k[c]), s.phi0[c]);
    trial[c] = fma(step, double(n.t[c]), s.phi0[c]);
  }
  const double dS = local_action<double, N>(trial, s.F, two_kappa, lambda) -
                    local_action<double, N>(phi, s.F, two_kappa, lambda);
  return dS <= 0.0 || u01<double>(aw) < q_exp(-dS);
}

// The hits of one FP64 site visit without FP64 arithmetic in the loop (an FP64
// instruction takes a warp 64 cycles; a hit took about 50 of them).  A proposal
// moves phi by delta (2u - 1) = delta 2^-23 k with an odd integer k, so accepted
// moves are summed as integers, and the new phi is phi0 + delta 2^-23 K, rounded
// once (in place of once per accepted hit).  The test u < exp(-dS) is decided
// in FP32 where its error bound allows:
//   dS = -2 kappa e.F + q (1 + lambda (2 P + q - 2)),  e = trial - phi,
//   q = e.(phi + trial), P = phi.phi;
// with W_c = 2 (|phi_c| + |phi0_c| + delta), which bounds |phi_c| + |trial_c| and,
// times 1.5 2^-24, the error of either, the roundings of 2^-24 add up to less than
// 16 2^-24 of
//   2 kappa a1 + a2 (1 + lambda (2 P + 2 + a2)) + lambda |q| sum W^2,
//   a1 = sum |e F|, a2 = sum |e| W (absolute values throughout),
// eps below; exp adds (4 + 2 |dS|) 2^-23.  Otherwise the test is taken in FP64.
// Infinities and NaN fail both comparisons and go there too.
template <int N>
struct OnHitsF64 {
  OnSite64 site;
  double two_kappa, lambda, step;
  float p0[4], p[4], F[4], W[4], kf, lf, sf, df, P, w2;
  int K[4];
  __device__ __forceinline__ OnHitsF64(const OnCtx& a, const double phi[4], const double f[4])
      : two_kappa(2.0 * a.kappa), lambda(a.lambda), step(a.delta * 0x1p-23) {
    kf = a.kf;
    lf = float(lambda);
    sf = float(step);
    df = fabsf(float(a.delta));
#pragma unroll
    for (int c = 0; c < 4; ++c) {
      site.phi0[c] = phi[c];
      site.F[c] = f[c];
      F[c] = float(f[c]);
    }
    restart();
  }
  __device__ __forceinline__ void restart() {
#pragma unroll
    for (int c = 0; c < N; ++c) {
      K[c] = 0;
      p0[c] = p[c] = float(site.phi0[c]);
    }
    bound();
  }
  __device__ __forceinline__ void bound() {
    w2 = 0.f;
    P = 0.f;
#pragma unroll
    for (int c = 0; c < N; ++c) {
      W[c] = 2.f * (fabsf(p[c]) + (fabsf(p0[c]) + df));
      w2 = fmaf(W[c], W[c], w2);
      P = fmaf(p[c], p[c], P);
    }
  }
  __device__ __forceinline__ bool hit(const uint4& w, uint32_t aw) {
    const uint32_t wu[4] = {w.x, w.y, w.z, w.w};
    float t[4], s1 = 0.f, q = 0.f, a1 = 0.f, a2 = 0.f;
    int T[4];
#pragma unroll
    for (int c = 0; c < N; ++c) {
      const int k = int((wu[c] >> 8) | 1u) - (1 << 23);
      T[c] = K[c] + k;
      t[c] = fmaf(sf, float(T[c]), p0[c]);
      const float e = sf * float(k);
      s1 = fmaf(e, F[c], s1);
      q = fmaf(e, p[c] + t[c], q);
      a1 = fmaf(fabsf(e), fabsf(F[c]), a1);
      a2 = fmaf(fabsf(e), W[c], a2);
    }
    const float x = fmaf(kf, s1, -q * fmaf(lf, fmaf(2.f, P, q) - 2.f, 1.f));
    const float E = __expf(x), u = u01<float>(aw);
    const float l = fabsf(lf);
    const float eps = 0x1p-20f * (fabsf(kf) * a1 + fmaf(a2, fmaf(l, fmaf(2.f, P, a2) + 2.f, 1.f), l * fabsf(q) * w2));
    const float m = fmaf(fabsf(x), 0x1p-22f, fmaf(2.f, eps, 0x1p-21f));
    bool yes = u < fmaf(-E, m, E);
    if (!yes && !(eps < 1.f && u > fmaf(E, m, E))) {
      OnSteps n;
#pragma unroll
      for (int c = 0; c < 4; ++c) {
        n.k[c] = c < N ? K[c] : 0;
        n.t[c] = c < N ? T[c] : 0;
      }
      yes = on_test_fp64<N>(site, n, two_kappa, lambda, step, aw);
    }
    if (!yes) return false;
#pragma unroll
    for (int c = 0; c < N; ++c) {
      K[c] = T[c];
      p[c] = t[c];
    }
    bound();
    return true;
  }
  // Every 128 hits at most: |K| stays below 2^30.
  __device__ __forceinline__ void flush() {
#pragma unroll
    for (int c = 0; c < N; ++c) site.phi0[c] = fma(step, double(K[c]), site.phi0[c]);
    restart();
  }
};

template <typename R, int N>
struct OnHits;
template <int N>
struct OnHits<float, N> : OnHitsF32<N> {
  using OnHitsF32<N>::OnHitsF32;
  __device__ __forceinline__ void result(float v[4]) const {
#pragma unroll
    for (int c = 0; c < 4; ++c) v[c] = this->phi[c];
  }
};
template <int N>
struct OnHits<double, N> : OnHitsF64<N> {
  using OnHitsF64<N>::OnHitsF64;
  __device__ __forceinline__ void result(double v[4]) const {
#pragma unroll
    for (int c = 0; c < 4; ++c) v[c] = this->site.phi0[c];
  }
};

// Blocks of up to 512 threads have to launch: 128 registers at most.  A sweep of
// O(4) with 100 hits per site, us, before -> now: FP32 8^3x8 55.9 -> 49.8, 32^4
// 456 -> 447 (80 registers; 64: 473, 128: 452); FP64 8^3x8 363 -> 81, 16^4 655 ->
// 101, 32^4 8649 -> 822.  Bound: the integer pipe (1.25 Philox blocks per hit, 160
// cycles of an SM sub-partition per warp and hit in FP32), at small sizes the
// latency of one hit after another.
constexpr int ON_MAXNREG_F32 = 80, ON_MAXNREG_F64 = 128;
template <typename R, int N>
__global__ void __maxnreg__(sizeof(R) == 4 ? ON_MAXNREG_F32 : ON_MAXNREG_F64) on_phase_kernel(const OnCtx a, int parity) {
  const int h = blockIdx.x * blockDim.x + threadIdx.x;
  unsigned n_acc = 0;
  if (h < a.g.Vh) {
    const Site sc = site_of(a.g, parity, h);
    LexSite x;
    x.c[0] = sc.x;
    x.c[1] = sc.y;
    x.c[2] = sc.z;
    x.c[3] = sc.t;
    x.s = 2 * h + (sc.x & 1);
    R F[4] = {R(0), R(0), R(0), R(0)};
    add_neighbours<R, 0>(a, parity ^ 1, x, F);
    add_neighbours<R, 1>(a, parity ^ 1, x, F);
    add_neighbours<R, 2>(a, parity ^ 1, x, F);
    add_neighbours<R, 3>(a, parity ^ 1, x, F);
    R phi[4];
    OnStore<R>::load(a, parity, h, phi);
    OnHits<R, N> site(a, phi, F);
    const uint32_t sweep = *a.sweep;
    // Four hits share an acceptance block; their four proposal blocks are drawn
    // with it, five independent Philox chains in flight.
    for (int hit = 0; hit < a.nhit; hit += 4) {
      const uint4 acc =
          philox4x32_10(make_uint4(uint32_t(x.s), sweep, KIND_ON_ACCEPT << 4, uint32_t(hit >> 2)), a.k0, a.k1);
      uint4 w[4];
#pragma unroll
      for (int j = 0; j < 4; ++j)
        w[j] = philox4x32_10(make_uint4(uint32_t(x.s), sweep, KIND_ON_PROPOSE << 4, uint32_t(hit + j)), a.k0, a.k1);
      const uint32_t aw[4] = {acc.x, acc.y, acc.z, acc.w};
      if (hit + 4 <= a.nhit) {
#pragma unroll
        for (int j = 0; j < 4; ++j) n_acc += site.hit(w[j], aw[j]);
      } else {
#pragma unroll
        for (int j = 0; j < 3; ++j)
          if (hit + j < a.nhit) n_acc += site.hit(w[j], aw[j]);
      }
      if ((hit & 127) == 124) site.flush();
    }
    site.flush();
    site.result(phi);
    OnStore<R>::store(a, parity, h, phi);
  }
  // one atomic per warp for the acceptance count
  const unsigned total = __reduce_add_sync(0xffffffffu, n_acc);
  if ((threadIdx.x & 31) == 0 && total) atomicAdd(a.accepted, (unsigned long long)total);
}

__global__ void on_advance_kernel(const OnCtx a) { *a.sweep_rw += 1u; }

template <typename R>
__global__ void on_start_kernel(const OnCtx a, int hot) {
  const int64_t idx = int64_t(blockIdx.x) * blockDim.x + threadIdx.x;
  if (idx >= 2LL * a.g.Vh) return;
  const int par = int(idx / a.g.Vh), h = int(idx % a.g.Vh);
  const Site x = site_of(a.g, par, h);
  const uint32_t s = uint32_t(lex(a.g, x));
  R v[4] = {R(0), R(0), R(0), R(0)};
  if (hot) {
    const uint4 w = philox4x32_10(make_uint4(s, 0xFFFFFFFFu, KIND_ON_START << 4, 0u), a.k0, a.k1);
    const uint32_t wu[4] = {w.x, w.y, w.z, w.w};
    for (int c = 0; c < a.N; ++c) v[c] = R(2.0 * u01<double>(wu[c]) - 1.0);
  } else {
    v[0] = R(1);
  }
  OnStore<R>::store(a, par, h, v);
}

// Canonical host order [s][c] (N doubles per site) <-> device layout.
template <typename R>
__global__ void on_to_canonical(const OnCtx a, double* out) {
  const int64_t idx = int64_t(blockIdx.x) * blockDim.x + threadIdx.x;
  if (idx >= 2LL * a.g.Vh) return;
  const int par = int(idx / a.g.Vh), h = int(idx % a.g.Vh);
  const int64_t s = lex(a.g, site_of(a.g, par, h));
  R v[4];
  OnStore<R>::load(a, par, h, v);
  for (int c = 0; c < a.N; ++c) out[s * a.N + c] = double(v[c]);
}

template <typename R>
__global__ void on_from_canonical(const OnCtx a, const double* in) {
  const int64_t idx = int64_t(blockIdx.x) * blockDim.x + threadIdx.x;
  if (idx >= 2LL * a.g.Vh) return;
  const int par = int(idx / a.g.Vh), h = int(idx % a.g.Vh);
  const int64_t s = lex(a.g, site_of(a.g, par, h));
  R v[4] = {R(0), R(0), R(0), R(0)};
  for (int c = 0; c < a.N; ++c) v[c] = R(in[s * a.N + c]);
  OnStore<R>::store(a, par, h, v);
}

// Per-site phi.phi, forward hopping term sum_mu phi_x.phi_{x+mu}, and phi_x,
// in the storage precision per site and FP64 across sites: per-block partials
// in a fixed order, then one block sums the partials in a fixed order.
template <typename R>
__global__ void __launch_bounds__(ON_MEAS_THREADS) on_measure_kernel(const OnCtx a) {
  const int64_t idx = int64_t(blockIdx.x) * ON_MEAS_THREADS + threadIdx.x;
  double v[ON_MEAS_VALUES] = {0.0, 0.0, 0.0, 0.0, 0.0, 0.0};
  if (idx < 2LL * a.g.Vh) {
    const int par = int(idx / a.g.Vh), h = int(idx % a.g.Vh);
    const Site x = site_of(a.g, par, h);
    R p[4];
    OnStore<R>::load(a, par, h, p);
    R pp = R(0), hop = R(0);
#pragma unroll
    for (int c = 0; c < 4; ++c) pp = fma(p[c], p[c], pp);
#pragma unroll
    for (int mu = 0; mu < 4; ++mu) {
      const Site y = step(a.g, x, mu, +1);
      R q[4];
      OnStore<R>::load(a, par ^ 1, lex(a.g, y) >> 1, q);
#pragma unroll
      for (int c = 0; c < 4; ++c) hop = fma(p[c], q[c], hop);
    }
    v[0] = double(pp);
    v[1] = double(hop);
#pragma unroll
    for (int c = 0; c < 4; ++c) v[2 + c] = double(p[c]);
  }
  __shared__ double sh[ON_MEAS_VALUES][ON_MEAS_THREADS];
#pragma unroll
  for (int k = 0; k < ON_MEAS_VALUES; ++k) sh[k][threadIdx.x] = v[k];
  __syncthreads();
  for (int w = ON_MEAS_THREADS / 2; w > 0; w >>= 1) {
    if (int(threadIdx.x) < w)
#pragma unroll
      for (int k = 0; k < ON_MEAS_VALUES; ++k) sh[k][threadIdx.x] += sh[k][threadIdx.x + w];
    __syncthreads();
  }
  if (threadIdx.x < ON_MEAS_VALUES) a.partials[ON_MEAS_VALUES * blockIdx.x + threadIdx.x] = sh[threadIdx.x][0];
}

__global__ void __launch_bounds__(1024) on_measure_final(const OnCtx a, int n_blocks) {
  __shared__ double sh[ON_MEAS_VALUES][1024];
  double s[ON_MEAS_VALUES] = {0.0, 0.0, 0.0, 0.0, 0.0, 0.0};
  for (int b = threadIdx.x; b < n_blocks; b += 1024)
#pragma unroll
    for (int k = 0; k < ON_MEAS_VALUES; ++k) s[k] += a.partials[ON_MEAS_VALUES * b + k];
#pragma unroll
  for (int k = 0; k < ON_MEAS_VALUES; ++k) sh[k][threadIdx.x] = s[k];
  __syncthreads();
  for (int w = 512; w > 0; w >>= 1) {
    if (int(threadIdx.x) < w)
#pragma unroll
      for (int k = 0; k < ON_MEAS_VALUES; ++k) sh[k][threadIdx.x] += sh[k][threadIdx.x + w];
    __syncthreads();
  }
  if (threadIdx.x == 0) {
    const double V = 2.0 * double(a.g.Vh);
    a.meas_out[0] = sh[0][0] / V;
    a.meas_out[1] = sh[1][0] / (4.0 * V);
    double m2 = 0.0;
    for (int c = 0; c < 4; ++c) {
      const double m = sh[2 + c][0] / V;
      a.meas_out[3 + c] = m;
      m2 += m * m;
    }
    a.meas_out[2] = sqrt(m2);
  }
}

template <typename R>
cudaError_t launch_on_phase(const OnCtx& a, int parity, int block, cudaStream_t st) {
  const unsigned grid = unsigned((a.g.Vh + block - 1) / block);
  switch (a.N) {
    case 1: on_phase_kernel<R, 1><<<grid, block, 0, st>>>(a, parity); break;
    case 2: on_phase_kernel<R, 2><<<grid, block, 0, st>>>(a, parity); break;
    case 3: on_phase_kernel<R, 3><<<grid, block, 0, st>>>(a, parity); break;
    default: on_phase_kernel<R, 4><<<grid, block, 0, st>>>(a, parity); break;
  }
  return cudaGetLastError();
}

thread_local char g_msg[512];

int fail(int code, const char* fmt, ...) {
  va_list ap;
  va_start(ap, fmt);
  vsnprintf(g_msg, sizeof g_msg, fmt, ap);
  va_end(ap);
  return set_last_error(code, g_msg);
}

}  // namespace
}  // namespace qcd

using namespace qcd;

struct qcd_on {
  int N = 0, Ns = 0, Nt = 0, precision = 0, nhit = 100, block = 128;
  double kappa = 0.0, lambda = 0.0, delta = 1.0;
  uint64_t seed = 0;
  cudaStream_t stream = nullptr;
  GeomH g{};
  void* phi = nullptr;
  unsigned char* d_small = nullptr;  // sweep counter, accepted hits, results
  double* d_partials = nullptr;
  int n_meas_blocks = 0;
  cudaGraphExec_t graph = nullptr;  // one sweep, for (graph_seed, nhit, block)
  uint64_t graph_seed = 0;
  int graph_nhit = 0, graph_block = 0;
};

namespace {

OnCtx make_on_ctx(const qcd_on* L, uint64_t seed) {
  OnCtx a{};
  a.phi = L->phi;
  a.g = L->g;
  a.N = L->N;
  a.nhit = L->nhit;
  a.kappa = L->kappa;
  // With steps or couplings this far from 1, underflow in FP32 could outgrow the
  // test's bound of roundings.
  a.kf = L->delta > 0x1p-60 && std::fabs(L->kappa) < 0x1p60 && std::fabs(L->lambda) < 0x1p60
             ? float(2.0 * L->kappa)
             : std::numeric_limits<float>::quiet_NaN();
  a.lambda = L->lambda;
  a.delta = L->delta;
  a.k0 = uint32_t(seed);  // lattice id 0
  a.k1 = uint32_t(seed >> 32);
  a.sweep = reinterpret_cast<const uint32_t*>(L->d_small);
  a.sweep_rw = reinterpret_cast<uint32_t*>(L->d_small);
  a.accepted = reinterpret_cast<unsigned long long*>(L->d_small + 8);
  a.partials = L->d_partials;
  a.meas_out = reinterpret_cast<double*>(L->d_small + 64);
  return a;
}

cudaError_t on_phase_launch(const qcd_on* L, int parity, uint64_t seed) {
  const OnCtx a = make_on_ctx(L, seed);
  return L->precision == QCD_FP64_PLAIN ? launch_on_phase<double>(a, parity, L->block, L->stream)
                                        : launch_on_phase<float>(a, parity, L->block, L->stream);
}

int check(const qcd_on* L) { return L ? QCD_OK : fail(QCD_ERR_INVALID_ARG, "null O(N) handle"); }

void drop_graph(qcd_on* L) {
  if (L->graph) cudaGraphExecDestroy(L->graph);
  L->graph = nullptr;
}

int build_graph(qcd_on* L, uint64_t seed) {
  drop_graph(L);
  cudaStream_t cap;
  if (cudaStreamCreateWithFlags(&cap, cudaStreamNonBlocking) != cudaSuccess)
    return fail(QCD_ERR_CUDA, "O(N) graph: stream creation failed");
  cudaGraph_t g = nullptr;
  cudaError_t e = cudaStreamBeginCapture(cap, cudaStreamCaptureModeThreadLocal);
  if (e == cudaSuccess) {
    qcd_on tmp = *L;
    tmp.stream = cap;
    const OnCtx a = make_on_ctx(&tmp, seed);
    cudaError_t e1 = on_phase_launch(&tmp, 0, seed);
    cudaError_t e2 = on_phase_launch(&tmp, 1, seed);
    on_advance_kernel<<<1, 1, 0, cap>>>(a);
    cudaError_t e3 = cudaGetLastError();
    e = cudaStreamEndCapture(cap, &g);
    if (e == cudaSuccess) e = e1 != cudaSuccess ? e1 : e2 != cudaSuccess ? e2 : e3;
  }
  if (e == cudaSuccess) e = cudaGraphInstantiate(&L->graph, g, 0);
  if (g) cudaGraphDestroy(g);
  cudaStreamDestroy(cap);
  if (e != cudaSuccess) {
    L->graph = nullptr;
    cudaGetLastError();
    return fail(QCD_ERR_CUDA, "O(N) graph: %s", cudaGetErrorString(e));
  }
  L->graph_seed = seed;
  L->graph_nhit = L->nhit;
  L->graph_block = L->block;
  return QCD_OK;
}

template <typename F>
int copy_via_device(qcd_on* L, size_t bytes, F&& body) {
  double* d = nullptr;
  cudaError_t e = cudaMallocAsync(reinterpret_cast<void**>(&d), bytes, L->stream);
  if (e != cudaSuccess) return fail(QCD_ERR_OOM, "O(N): %zu bytes of staging: %s", bytes, cudaGetErrorString(e));
  e = body(d);
  cudaFreeAsync(d, L->stream);
  const cudaError_t e2 = cudaStreamSynchronize(L->stream);
  if (e == cudaSuccess) e = e2;
  return e == cudaSuccess ? QCD_OK : fail(QCD_ERR_CUDA, "O(N) field copy: %s", cudaGetErrorString(e));
}

}  // namespace

extern "C" {

int qcd_on_create(qcd_on** out, int N, int Ns, int Nt, double kappa, double lambda, double delta, int precision,
                  int start, uint64_t seed, void* stream) {
  if (!out) return fail(QCD_ERR_INVALID_ARG, "out is null");
  *out = nullptr;
  if (N < 1 || N > 4) return fail(QCD_ERR_INVALID_ARG, "N must be 1..4, got %d", N);
  if (Ns < 2 || Nt < 2 || (Ns & 1) || (Nt & 1))
    return fail(QCD_ERR_INVALID_ARG, "Ns and Nt must be even and >= 2 (got %d, %d)", Ns, Nt);
  const long long V = (long long)Ns * Ns * Ns * Nt;
  if (V >= (1LL << 31) || Ns > 1290) return fail(QCD_ERR_INVALID_ARG, "lattice too large (V = %lld)", V);
  if (!(delta > 0.0) || !(kappa == kappa) || !(lambda == lambda))
    return fail(QCD_ERR_INVALID_ARG, "delta must be > 0 and kappa, lambda finite");
  if (precision != QCD_FP64_PLAIN && precision != QCD_FP32_COMPRESSED)
    return fail(QCD_ERR_INVALID_ARG, "unknown precision %d", precision);
  if (start != QCD_COLD && start != QCD_HOT) return fail(QCD_ERR_INVALID_ARG, "unknown start %d", start);
  qcd_on* L = new (std::nothrow) qcd_on();
  if (!L) return fail(QCD_ERR_OOM, "host allocation failed");
  L->N = N;
  L->Ns = Ns;
  L->Nt = Nt;
  L->precision = precision;
  L->kappa = kappa;
  L->lambda = lambda;
  L->delta = delta;
  L->seed = seed;
  L->stream = static_cast<cudaStream_t>(stream);
  L->g.Ns = Ns;
  L->g.Nt = Nt;
  L->g.Vh = int(V / 2);
  geom_set_decode(L->g);
  L->g.plane = (L->g.Vh + 63) / 64 * 64;
  L->n_meas_blocks = int((V + ON_MEAS_THREADS - 1) / ON_MEAS_THREADS);
  const size_t field_bytes = size_t(2) * size_t(L->g.plane) * 16 * (precision == QCD_FP64_PLAIN ? 2 : 1);
  if (cudaMalloc(&L->phi, field_bytes) != cudaSuccess ||
      cudaMalloc(reinterpret_cast<void**>(&L->d_small), 256) != cudaSuccess ||
      cudaMalloc(reinterpret_cast<void**>(&L->d_partials), sizeof(double) * ON_MEAS_VALUES * L->n_meas_blocks) !=
          cudaSuccess) {
    cudaGetLastError();
    qcd_on_destroy(L);
    return fail(QCD_ERR_OOM, "device allocation of %zu bytes of field failed", field_bytes);
  }
  cudaError_t e = cudaMemsetAsync(L->d_small, 0, 256, L->stream);
  if (e == cudaSuccess) e = cudaMemsetAsync(L->phi, 0, field_bytes, L->stream);
  if (e == cudaSuccess) {
    const OnCtx a = make_on_ctx(L, seed);
    const unsigned grid = unsigned((V + 255) / 256);
    if (precision == QCD_FP64_PLAIN) on_start_kernel<double><<<grid, 256, 0, L->stream>>>(a, start);
    else on_start_kernel<float><<<grid, 256, 0, L->stream>>>(a, start);
    e = cudaGetLastError();
  }
  if (e == cudaSuccess) e = cudaStreamSynchronize(L->stream);
  if (e != cudaSuccess) {
    qcd_on_destroy(L);
    return fail(QCD_ERR_CUDA, "O(N) create: %s", cudaGetErrorString(e));
  }
  *out = L;
  return QCD_OK;
}

int qcd_on_destroy(qcd_on* L) {
  if (!L) return QCD_OK;
  if (L->stream) cudaStreamSynchronize(L->stream);
  else cudaDeviceSynchronize();
  drop_graph(L);
  cudaFree(L->phi);
  cudaFree(L->d_small);
  cudaFree(L->d_partials);
  delete L;
  return QCD_OK;
}

int qcd_on_set_nhit(qcd_on* L, int nhit) {
  if (int rc = check(L)) return rc;
  if (nhit < 1) return fail(QCD_ERR_INVALID_ARG, "nhit must be >= 1");
  L->nhit = nhit;
  return QCD_OK;
}

int qcd_on_set_block(qcd_on* L, int threads) {
  if (int rc = check(L)) return rc;
  if (threads != 64 && threads != 128 && threads != 256 && threads != 512)
    return fail(QCD_ERR_INVALID_ARG, "threads must be 64, 128, 256 or 512");
  L->block = threads;
  return QCD_OK;
}

int qcd_on_sweep(qcd_on* L, int n_sweeps, uint64_t seed) {
  if (int rc = check(L)) return rc;
  if (n_sweeps < 0) return fail(QCD_ERR_INVALID_ARG, "n_sweeps must be >= 0");
  if (n_sweeps == 0) return QCD_OK;
  if (!L->graph || L->graph_seed != seed || L->graph_nhit != L->nhit || L->graph_block != L->block)
    if (int rc = build_graph(L, seed)) return rc;
  for (int i = 0; i < n_sweeps; ++i) {
    const cudaError_t e = cudaGraphLaunch(L->graph, L->stream);
    if (e != cudaSuccess) return fail(QCD_ERR_CUDA, "O(N) sweep: %s", cudaGetErrorString(e));
  }
  return QCD_OK;
}

int qcd_on_phase(qcd_on* L, int parity, uint64_t seed) {
  if (int rc = check(L)) return rc;
  if (parity != 0 && parity != 1) return fail(QCD_ERR_INVALID_ARG, "parity must be 0 or 1");
  const cudaError_t e = on_phase_launch(L, parity, seed);
  return e == cudaSuccess ? QCD_OK : fail(QCD_ERR_CUDA, "O(N) phase: %s", cudaGetErrorString(e));
}

int qcd_on_measure(qcd_on* L, double* out) {
  if (int rc = check(L)) return rc;
  if (!out) return fail(QCD_ERR_INVALID_ARG, "out is null");
  const OnCtx a = make_on_ctx(L, L->seed);
  if (L->precision == QCD_FP64_PLAIN)
    on_measure_kernel<double><<<L->n_meas_blocks, ON_MEAS_THREADS, 0, L->stream>>>(a);
  else
    on_measure_kernel<float><<<L->n_meas_blocks, ON_MEAS_THREADS, 0, L->stream>>>(a);
  on_measure_final<<<1, 1024, 0, L->stream>>>(a, L->n_meas_blocks);
  cudaError_t e = cudaGetLastError();
  if (e == cudaSuccess) e = cudaMemcpyAsync(out, a.meas_out, 7 * sizeof(double), cudaMemcpyDeviceToHost, L->stream);
  if (e == cudaSuccess) e = cudaStreamSynchronize(L->stream);
  return e == cudaSuccess ? QCD_OK : fail(QCD_ERR_CUDA, "O(N) measure: %s", cudaGetErrorString(e));
}

int qcd_on_get_field(qcd_on* L, double* host_out) {
  if (int rc = check(L)) return rc;
  if (!host_out) return fail(QCD_ERR_INVALID_ARG, "host_out is null");
  const size_t bytes = size_t(2) * L->g.Vh * L->N * sizeof(double);
  return copy_via_device(L, bytes, [&](double* d) {
    const OnCtx a = make_on_ctx(L, L->seed);
    const unsigned grid = unsigned((2LL * L->g.Vh + 255) / 256);
    if (L->precision == QCD_FP64_PLAIN) on_to_canonical<double><<<grid, 256, 0, L->stream>>>(a, d);
    else on_to_canonical<float><<<grid, 256, 0, L->stream>>>(a, d);
    cudaError_t e = cudaGetLastError();
    if (e == cudaSuccess) e = cudaMemcpyAsync(host_out, d, bytes, cudaMemcpyDeviceToHost, L->stream);
    return e;
  });
}

int qcd_on_set_field(qcd_on* L, const double* host_in) {
  if (int rc = check(L)) return rc;
  if (!host_in) return fail(QCD_ERR_INVALID_ARG, "host_in is null");
  const size_t bytes = size_t(2) * L->g.Vh * L->N * sizeof(double);
  return copy_via_device(L, bytes, [&](double* d) {
    cudaError_t e = cudaMemcpyAsync(d, host_in, bytes, cudaMemcpyHostToDevice, L->stream);
    const OnCtx a = make_on_ctx(L, L->seed);
    const unsigned grid = unsigned((2LL * L->g.Vh + 255) / 256);
    if (e == cudaSuccess) {
      if (L->precision == QCD_FP64_PLAIN) on_from_canonical<double><<<grid, 256, 0, L->stream>>>(a, d);
      else on_from_canonical<float><<<grid, 256, 0, L->stream>>>(a, d);
      e = cudaGetLastError();
    }
    return e;
  });
}

int qcd_on_get_sweep(qcd_on* L, uint32_t* sweep) {
  if (int rc = check(L)) return rc;
  if (!sweep) return fail(QCD_ERR_INVALID_ARG, "sweep is null");
  cudaError_t e = cudaMemcpyAsync(sweep, L->d_small, sizeof(uint32_t), cudaMemcpyDeviceToHost, L->stream);
  if (e == cudaSuccess) e = cudaStreamSynchronize(L->stream);
  return e == cudaSuccess ? QCD_OK : fail(QCD_ERR_CUDA, "O(N) get_sweep: %s", cudaGetErrorString(e));
}

int qcd_on_set_sweep(qcd_on* L, uint32_t sweep) {
  if (int rc = check(L)) return rc;
  cudaError_t e = cudaMemcpyAsync(L->d_small, &sweep, sizeof(uint32_t), cudaMemcpyHostToDevice, L->stream);
  if (e == cudaSuccess) e = cudaStreamSynchronize(L->stream);
  return e == cudaSuccess ? QCD_OK : fail(QCD_ERR_CUDA, "O(N) set_sweep: %s", cudaGetErrorString(e));
}

int qcd_on_get_accepted(qcd_on* L, unsigned long long* accepted) {
  if (int rc = check(L)) return rc;
  if (!accepted) return fail(QCD_ERR_INVALID_ARG, "accepted is null");
  cudaError_t e =
      cudaMemcpyAsync(accepted, L->d_small + 8, sizeof(unsigned long long), cudaMemcpyDeviceToHost, L->stream);
  if (e == cudaSuccess) e = cudaStreamSynchronize(L->stream);
  return e == cudaSuccess ? QCD_OK : fail(QCD_ERR_CUDA, "O(N) get_accepted: %s", cudaGetErrorString(e));
}

}  // extern "C"
