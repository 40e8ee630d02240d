// qcd_fixmath.cuh -- the functions of the FP64 heat-bath draw in fixed point
// (qcd_fix.cuh): logarithm, cosine and sine of uniforms, square roots, and the
// Kennedy-Pendleton draw made of them.  In FP64 one draw is about 290
// instructions of 64 cycles; here it is about 800 of 2.
//
// Methods: the logarithm by a table of reciprocals of the leading 7 bits, whose
// product with the argument leaves an exact r (|r| < 2^-7.8) for the Taylor
// series of ln(1 + r); cosine and sine by a table of a quarter turn in 64 steps
// and the Taylor series of the remaining angle (at most pi/256); square roots by
// an approximate reciprocal square root and one step of third order.  Absolute
// errors are a few 2^-58, measured against the 64-bit mantissa's long double in
// the tests.
#pragma once

#include "qcd_fix.cuh"
#include "qcd_fixtab.h"
#ifdef __CUDACC__
#include "qcd_device.cuh"
#endif

namespace qcd {

#ifdef __CUDACC__
static __device__ const FxLogEntry fx_log_table[128] = {QCD_FX_LOG_TABLE};
static __device__ const FxTrigEntry fx_trig_table[65] = {QCD_FX_TRIG_TABLE};
#endif
#ifndef __CUDA_ARCH__
static const FxLogEntry fx_log_table_host[128] = {QCD_FX_LOG_TABLE};
static const FxTrigEntry fx_trig_table_host[65] = {QCD_FX_TRIG_TABLE};
#endif
QCD_HD FxLogEntry fx_log_entry(int i) {
#ifdef __CUDA_ARCH__
  const longlong2 v = __ldg(reinterpret_cast<const longlong2*>(fx_log_table) + i);
  return {v.x, v.y};
#else
  return fx_log_table_host[i];
#endif
}
QCD_HD FxTrigEntry fx_trig_entry(int j) {
#ifdef __CUDA_ARCH__
  const longlong2 v = __ldg(reinterpret_cast<const longlong2*>(fx_trig_table) + j);
  return {v.x, v.y};
#else
  return fx_trig_table_host[j];
#endif
}

QCD_HD int64_t fx_product(int64_t a, int64_t b) {
  FxAcc s;
  s.add(fx_limbs(a), fx_limbs(b));
  return s.value();
}

constexpr int64_t FX_ONE = int64_t(1) << FX_UNIT;
constexpr int64_t FX_LN2 = 199786072581291495;

// -ln(n 2^-24) = z ln 2 + g for an integer n in [1, 2^24): g in [0, ln 2].
QCD_HD void fx_neglog24(uint32_t n, int& z, int64_t& g) {
#ifdef __CUDA_ARCH__
  z = __clz(int(n)) - 8;
#else
  z = __builtin_clz(n) - 8;
#endif
  const uint32_t N = n << z;  // [2^23, 2^24)
  const FxLogEntry t = fx_log_entry((N >> 16) & 127);
  // r 2^33 = N c - 2^33, below 2^26 in magnitude: the low word is enough
  const int32_t r33 = int32_t(N * uint32_t(t.c));
  const int32_t R = int32_t(uint32_t(r33) << 5);  // r 2^38
  // ln(1 + r) = r - r^2 (1/2 - r (1/3 - r (1/4 - r (1/5 - r (1/6 - r / 7)))))
  int32_t p = 357913941 - int32_t(fx_mad(R, 306783378, 0) >> 38);  // 2^-31
  p = 429496730 - int32_t(fx_mad(R, p, 0) >> 38);
  p = 536870912 - int32_t(fx_mad(R, p, 0) >> 38);
  const int64_t p3 = 96076792050570581 - (fx_mad(R, p, 0) >> 11);
  const Fx l3 = fx_limbs(p3);
  const int64_t q = 144115188075855872 - ((fx_mad(R, l3.hi, 0) >> 9) + (fx_mad(R, l3.lo, 0) >> 38));
  const int64_t r2 = fx_mad(R, R, 0) >> 18;
  const int64_t ln1p = (int64_t(r33) << 25) - fx_product(r2, q);
  g = t.l - ln1p;
}

// Cosine and sine of x turns 2^-32.
QCD_HD void fx_sincos(uint32_t x, int64_t& c, int64_t& s) {
  const uint32_t y = x & 0x3fffffffu;
  const int j = int((y + (1u << 23)) >> 24);
  const int32_t d = int32_t(y) - (j << 24);
  const FxTrigEntry t = fx_trig_entry(j);
  // theta = d pi 2^-31: pi 2^27 = 2^-29 226375608064910089
  constexpr int64_t K = 226375608064910089;
  const int64_t th = fx_add(fx_mad(d, int32_t(K >> 29), 0), fx_mad(d, int32_t(K & FX_MASK), 0) >> 29);
  const Fx lt = fx_limbs(th);
  FxAcc sq;
  sq.add(lt, lt);
  const int64_t t2 = sq.value();
  const Fx l2 = fx_limbs(t2);
  auto times = [](const Fx& a, int64_t b) {
    FxAcc v;
    v.add(a, fx_limbs(b));
    return v.value();
  };
  // sin = th - th^3 (1/6 - th^2 (1/120 - th^2 / 5040))
  const int64_t w = 48038396025285291 - times(l2, 2401919801264265 - times(l2, 57188566696768));
  const int64_t sn = fx_sub(th, times(lt, times(l2, w)));
  // cos = 1 - th^2 / 2 + th^4 (1/24 - th^2 / 720)
  const int64_t cm = (t2 >> 1) - times(l2, times(l2, 12009599006321323 - times(l2, 400319966877377)));  // 1 - cos
  const Fx C = fx_limbs(t.c), S = fx_limbs(t.s), a = fx_limbs(sn), b = fx_limbs(cm);
  FxAcc p, q, u, v;
  p.add(S, a);
  p.add(C, b);
  u.add(C, a);
  v.add(S, b);
  const int64_t cc = fx_sub(t.c, p.value());
  const int64_t ss = fx_add(t.s, fx_diff(u, v));
  const uint32_t quadrant = x >> 30;
  c = (quadrant & 1) ? ss : cc;
  s = (quadrant & 1) ? cc : ss;
  if (quadrant == 1 || quadrant == 2) c = -c;
  if (quadrant >= 2) s = -s;
}

// 1 / sqrt(n) for n in [1/4, 4].  The seed y stays below 2 (it can round up to it at
// n = 1/4): y^2 has to fit two limbs, and one unit of 2^-27 is within the seed's error.
QCD_HD int64_t fx_rsqrt(int64_t n) {
  const Fx l = fx_limbs(n);
  const float f = float(l.hi > 0 ? l.hi : 1);  // n 2^29
#ifdef __CUDA_ARCH__
  const int32_t seed = __float2int_rn(rsqrtf(f) * 3109888511975.f);  // 2^41.5 / sqrt(n 2^29) = y 2^27
#else
  const int32_t seed = int32_t(3109888511975.f / std::sqrt(f) + 0.5f);
#endif
  const int32_t yi = seed < (1 << 28) ? seed : (1 << 28) - 1;
  const Fx y2 = fx_limbs(fx_mad(yi, yi, 0) << 4);
  FxAcc m;
  m.add(l, y2);
  const int64_t e = fx_sub(FX_ONE, m.value());
  const int32_t es = int32_t(e >> 18);
  const int64_t t = (e >> 1) + ((3 * fx_mad(es, es, 0)) >> 25);
  return (int64_t(yi) << 31) + ((int64_t(yi) * (t >> 2)) >> 25);
}

// sqrt(x) for x in [0, 4).
QCD_HD int64_t fx_sqrt(int64_t x) {
  if (x <= 0) return 0;
  const int k = (fx_clz(uint64_t(x)) - 5) >> 1;  // x 4^k in [1/2, 2)
  const int64_t n = k >= 0 ? int64_t(uint64_t(x) << (2 * k)) : x >> (-2 * k);
  const int64_t s = fx_product(n, fx_rsqrt(n));
  return k >= 0 ? s >> k : s << -k;
}

// One Kennedy-Pendleton try on the words of its Philox block (uniforms
// (m + 1/2) 2^-23, m the upper 23 bits): e = -ln u2 - ln u1 cos^2(2 pi u3), and
// u4^2 (e in 2^-57 units: it reaches 33.3; u4^2 in 2^-58).
QCD_HD uint32_t fx_odd24(uint32_t w) { return ((w >> 9) << 1) | 1u; }

QCD_HD int64_t fx_kp_e(uint32_t w0, uint32_t w1, uint32_t w2) {
  int z0, z1;
  int64_t g0, g1, c, s;
  fx_neglog24(fx_odd24(w0), z0, g0);
  fx_neglog24(fx_odd24(w1), z1, g1);
  fx_sincos(fx_odd24(w2) << 8, c, s);
  const int64_t c2 = fx_product(c, c);
  return (int64_t(z1) * (FX_LN2 >> 1) + int64_t(z0) * (fx_product(FX_LN2, c2) >> 1)) +
         ((g1 + fx_product(g0, c2)) >> 1);
}
QCD_HD int64_t fx_kp_a3(uint32_t w3) {
  const uint32_t n = fx_odd24(w3);
  return int64_t(uint64_t(n) * n) << 10;
}

// Whether an accepted try's e (2^-57 units) is too small for fixed point: fx_kp_e is
// right to about 2^-57, which the square root below magnifies; below 2^-16 (one
// draw in 22 million: an FP64 update takes its warp 100 us) the update is left to FP64,
// whose error is relative.
QCD_HD bool fx_kp_small(double e) { return uint32_t(fx_bits(e) >> 32) < uint32_t(1023 + FX_UNIT - 1 - 16) << 20; }
// delta = d 2^-57 of a try by the double's exponent and mantissa, m 2^(-63 - e) with m in
// [2^63, 2^64): a small delta (weak coupling) keeps its bits.  e is negative for
// delta >= 2, which no try accepts (infinities too).
struct FxDelta {
  uint64_t m;
  int e;
  QCD_HD explicit FxDelta(double d)
      : m((uint64_t(1) << 63) | (fx_bits(d) << 11)), e(1023 + FX_UNIT - 1 - int(fx_bits(d) >> 52)) {}
  QCD_HD int64_t value() const { return e >= 0 ? int64_t(fx_shr(m, 5u + uint32_t(e))) : 4 * FX_ONE; }
  // sqrt(delta (2 - delta)) by delta 4^k in [1/2, 2).
  QCD_HD int64_t modulus(int64_t delta) const {
    const int64_t s = fx_sqrt(fx_product(int64_t(m >> (5 + (e & 1))), 2 * FX_ONE - delta));
    return int64_t(fx_shr(uint64_t(s), uint32_t(e) >> 1));
  }
};

// The unit vector of the direction block: (sin th cos ph, sin th sin ph, cos th)
// with cos th = 2 u0 - 1, ph = 2 pi u1.
QCD_HD void fx_direction(uint32_t w0, uint32_t w1, int64_t d[3]) {
  const uint32_t n = fx_odd24(w0);
  int64_t c, s;
  fx_sincos(fx_odd24(w1) << 8, c, s);
  // 4 u (1 - u) = n (2^24 - n) 2^-46
  const int64_t st = fx_sqrt(int64_t(uint64_t(n) * ((1u << 24) - n)) << 12);
  d[0] = fx_product(st, c);
  d[1] = fx_product(st, s);
  d[2] = (int64_t(n) << 35) - FX_ONE;
}

// a b of quaternions (matrix product, as qmul).
QCD_HD void fx_qmul(const Fx a[4], const Fx b[4], int64_t c[4]) {
  const Fx n1 = fx_neg(a[1]), n2 = fx_neg(a[2]), n3 = fx_neg(a[3]);
  FxAcc s0, s1, s2, s3;
  s0.add(a[0], b[0]);
  s0.add(n1, b[1]);
  s0.add(n2, b[2]);
  s0.add(n3, b[3]);
  s1.add(a[0], b[1]);
  s1.add(a[1], b[0]);
  s1.add(n2, b[3]);
  s1.add(a[3], b[2]);
  s2.add(a[0], b[2]);
  s2.add(a[2], b[0]);
  s2.add(n3, b[1]);
  s2.add(a[1], b[3]);
  s3.add(a[0], b[3]);
  s3.add(a[3], b[0]);
  s3.add(n1, b[2]);
  s3.add(a[2], b[1]);
  c[0] = s0.value();
  c[1] = s1.value();
  c[2] = s2.value();
  c[3] = s3.value();
}

#ifdef __CUDACC__
// What does not depend on the weight: try 0 and the direction.
struct FxKpFirst {
  double e;
  int64_t a3, d[3];
};
__device__ __forceinline__ FxKpFirst fx_kp_first(const Stream& tries, const Stream& dir) {
  FxKpFirst f;
  const uint4 w = philox4x32_10(make_uint4(tries.c0, tries.c1, tries.c2, 0u), tries.k0, tries.k1);
  f.e = double(fx_kp_e(w.x, w.y, w.z));
  f.a3 = fx_kp_a3(w.w);
  const uint4 v = philox4x32_10(make_uint4(dir.c0, dir.c1, dir.c2, 0u), dir.k0, dir.k1);
  fx_direction(v.x, v.y, f.d);
  return f;
}

// Heat-bath draw for the weight exp(alpha X0) with alpha = scale |w|, w != 0 in
// 2^-58 units and inv_scale = 1 / scale: r = X (w / |w|)^+.  Says when all nhit tries
// fail, or the draw is one for FP64 (r then holds it to less).  The ranges that alpha
// may have (any beta) are FP64's, so 1 / alpha and delta = e / alpha are formed there
// (three FP64 instructions); the test and all that follows are fixed point again.
// Error of the drawn quaternion against long double, largest / rms, in units of that
// of the same expressions in double: 0.39 / 0.36 at alpha = 3, 0.97 / 0.20 at 10,
// 0.76 / 0.18 at 100, 0.46 / 0.16 at 1e4 (with delta in 2^-58 units throughout and no
// bound on e: 0.39 / 0.36, 0.9 / 0.20, 6.4 / 0.4, 190 / 5 over 2 million draws, and
// 5, 52, 340, 16000 for e next to 0).
enum { FX_DRAWN = 0, FX_EXHAUSTED = 1, FX_SMALL_DRAW = 2 };
__device__ __forceinline__ int fx_heatbath(int64_t w[4], double inv_scale, int nhit, const Stream& tries,
                                            const FxKpFirst& f, Fx r[4]) {
  const int shift = fx_clz(fx_size4(w)) - 6;  // |w| = |w 2^shift| 2^-shift
  fx_normalise4(w);
  Fx v[4];
  FxAcc n;
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    v[k] = fx_limbs(w[k]);
    n.add(v[k], v[k]);
  }
  const int64_t rk = fx_rsqrt(n.value());
  const double inv_alpha =
      __hiloint2double(__double2hiint(fx_double(rk)) + (shift << 20), __double2loint(fx_double(rk))) * inv_scale;
  int64_t a3 = f.a3, delta;
  double e = f.e;
  FxDelta fd(0.0);
  bool drawn;
  for (int t = 0;;) {
    fd = FxDelta(e * inv_alpha);
    delta = fd.value();
    drawn = delta <= 2 * FX_ONE - 2 * a3;
    if (drawn || ++t >= nhit) break;
    const uint4 u = philox4x32_10(make_uint4(tries.c0, tries.c1, tries.c2, uint32_t(t)), tries.k0, tries.k1);
    e = double(fx_kp_e(u.x, u.y, u.z));
    a3 = fx_kp_a3(u.w);
  }
  const Fx lm = fx_limbs(fd.modulus(delta));
  const Fx lr = fx_limbs(rk);
  Fx X[4] = {fx_limbs(FX_ONE - delta)};
  Fx b[4];
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    FxAcc s;
    s.add(v[k], lr);
    b[k] = fx_limbs(k ? -s.value() : s.value());
    if (k) {
      FxAcc q;
      q.add(lm, fx_limbs(f.d[k - 1]));
      X[k] = fx_limbs(q.value());
    }
  }
  int64_t c[4];
  fx_qmul(X, b, c);
#pragma unroll
  for (int k = 0; k < 4; ++k) r[k] = fx_limbs(c[k]);
  return !drawn ? FX_EXHAUSTED : fx_kp_small(e) ? FX_SMALL_DRAW : FX_DRAWN;
}
#endif

}  // namespace qcd
