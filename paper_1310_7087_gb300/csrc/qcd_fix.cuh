// qcd_fix.cuh -- fixed-point complex arithmetic for FP64-stored links.
//
// One FP64 instruction of a warp occupies this GPU's FP64 unit for 64 cycles of
// an SM sub-partition (2 lanes per clock and SM); so does every conversion to or
// from FP64.  A 32 x 32 -> 64 bit integer multiply-add takes 2.  Link elements
// and their products are bounded by 1, so they need no exponent: a real v is
// held as the integer v 2^58 in two limbs, hi 2^29 + lo, and a multiply-add is
// three integer multiply-adds, hi hi' into one 64-bit accumulator and
// hi lo' + lo hi' into another (6 cycles).  Dropped: lo lo' (below 2^-58).
//
// Error: 2^-58 absolute per quantised input and per product sum, against the
// 2^-54 of each FP64 rounding of a number in [1/2, 1); sums of products are
// exact between the two.  (fx_load_int rounds towards zero and value() down, so the
// errors have a sign, a sixteenth of the rounding that storing a result adds.)
//
// Ranges, above: for |v| < 2 a limb product is below 2^60 (hi hi') or 2^59 (hi lo'),
// so a three-term complex dot product (6 real products per part, 12 cross
// terms) stays below 2^62.6 in both accumulators.  fx_load reports the largest
// exponent it saw and fx_check any result outside [-2, 2); a caller that finds
// one (infinities and NaN among them) takes its FP64 path.  Below: a few 2^-58 are
// less than FP64's rounding of numbers of order 1 only, so a staple sum, a subgroup
// block, a link or a product whose parts are all small (fx_small, fx_small_block,
// fx_tiny: links that are scaled down, next to never a sum that cancels) is left to
// FP64 too.
//
// Plain C++ besides a few device instructions, so that the host
// compiler can run the same arithmetic.
#pragma once

#include <cmath>
#include <cstdint>
#include <cstring>

#ifdef __CUDACC__
#define QCD_HD __host__ __device__ __forceinline__
#else
#define QCD_HD inline
#endif

namespace qcd {

constexpr int FX_UNIT = 58;  // v 2^58
constexpr int FX_LIMB = 29;
constexpr int32_t FX_MASK = (1 << FX_LIMB) - 1;

struct Fx {
  int32_t hi, lo;
};
struct FxC {
  Fx re, im;
};

// c + a b
QCD_HD int64_t fx_mad(int32_t a, int32_t b, int64_t c) {
#ifdef __CUDA_ARCH__
  int64_t r;
  asm("mad.wide.s32 %0, %1, %2, %3;" : "=l"(r) : "r"(a), "r"(b), "l"(c));
  return r;
#else
  return int64_t(uint64_t(c) + uint64_t(int64_t(a) * b));
#endif
}
// v >> s, 0 for s > 63 (PTX clamps the shift)
QCD_HD uint64_t fx_shr(uint64_t v, uint32_t s) {
#ifdef __CUDA_ARCH__
  uint64_t r;
  asm("shr.u64 %0, %1, %2;" : "=l"(r) : "l"(v), "r"(s));
  return r;
#else
  return s > 63 ? 0 : v >> s;
#endif
}
// wrapping sums (a caller that overflows has been told so by fx_check)
QCD_HD int64_t fx_add(int64_t a, int64_t b) { return int64_t(uint64_t(a) + uint64_t(b)); }
QCD_HD int64_t fx_sub(int64_t a, int64_t b) { return int64_t(uint64_t(a) - uint64_t(b)); }

QCD_HD uint64_t fx_bits(double x) {
#ifdef __CUDA_ARCH__
  return uint64_t(__double_as_longlong(x));
#else
  uint64_t b;
  std::memcpy(&b, &x, 8);
  return b;
#endif
}
QCD_HD double fx_real(uint64_t b) {
#ifdef __CUDA_ARCH__
  return __longlong_as_double(int64_t(b));
#else
  double x;
  std::memcpy(&x, &b, 8);
  return x;
#endif
}

// x to fixed point.  `big` collects the upper words: an exponent of 2 or more
// (infinity and NaN too) sets bit 30.  On the device one conversion on the FP64
// unit, which the integer arithmetic leaves idle, after the scaling by 2^58 as an
// addition to the exponent.
QCD_HD Fx fx_load(double x, uint32_t& big) {
  const uint64_t b = fx_bits(x);
  big |= uint32_t(b >> 32);
#ifdef __CUDA_ARCH__
  const int64_t r = __double2ll_rn(fx_real(b + (uint64_t(FX_UNIT) << 52)));
  return {int32_t(r >> FX_LIMB), int32_t(r) & FX_MASK};
#else
  const double v = x * 288230376151711744.0;
  const int64_t r = v > -9.2e18 && v < 9.2e18 ? int64_t(std::nearbyint(v)) : 0;
  return {int32_t(r >> FX_LIMB), int32_t(r) & FX_MASK};
#endif
}
// The same by integer instructions (14 against 5, but no FP64 unit to queue
// for): the mantissa shifted by its exponent to units of 2^-61, whose upper word
// is the high limb.  Towards zero.
QCD_HD Fx fx_load_int(double x, uint32_t& big) {
  const uint64_t b = fx_bits(x);
  const uint32_t hw = uint32_t(b >> 32), lw = uint32_t(b);
  big |= hw;
  const uint64_t m = (uint64_t((hw << 11) | (lw >> 21) | 0x80000000u) << 32) | (lw << 11);
  const uint64_t v = fx_shr(m, 1025u - ((hw >> 20) & 0x7ffu));
  Fx r{int32_t(v >> 32), int32_t(uint32_t(v) >> 3)};
  if (int32_t(hw) < 0) {
    r.hi = -r.hi;
    r.lo = -r.lo;
  }
  return r;
}
constexpr uint32_t FX_BIG = 0x40000000u, FX_BAD = 0xF0000000u;

QCD_HD Fx fx_limbs(int64_t r) { return {int32_t(r >> FX_LIMB), int32_t(r) & FX_MASK}; }
QCD_HD int64_t fx_value(Fx a) { return int64_t(uint64_t(int64_t(a.hi)) << FX_LIMB) + a.lo; }

// r 2^-58, rounded to nearest
QCD_HD double fx_double(int64_t r) {
  const uint64_t b = fx_bits(double(r));
  return fx_real(r ? b - (uint64_t(FX_UNIT) << 52) : b);
}

// Remembers in `bad` (bits 28 to 31) whether r is outside [-2, 2).
QCD_HD void fx_check(int64_t r, uint32_t& bad) {
  bad |= uint32_t(uint64_t(r) >> 32) + (1u << 27);
}

// sum of products: h counts 2^-58, m counts 2^-87
struct FxAcc {
  int64_t h = 0, m = 0;
  QCD_HD void add(Fx a, Fx b) {
    h = fx_mad(a.hi, b.hi, h);
    m = fx_mad(a.hi, b.lo, m);
    m = fx_mad(a.lo, b.hi, m);
  }
  QCD_HD int64_t value() const { return fx_add(h, m >> FX_LIMB); }
};
QCD_HD int64_t fx_diff(const FxAcc& p, const FxAcc& q) {
  return fx_add(fx_sub(p.h, q.h), fx_sub(p.m, q.m) >> FX_LIMB);
}

// sum a_k b_k, or with CONJ sum a_k conj(b_k)
template <bool CONJ>
struct FxDot {
  FxAcc s, p, q;
  QCD_HD void add(const FxC& a, const FxC& b) {
    if (CONJ) {
      s.add(a.re, b.re);
      s.add(a.im, b.im);
      p.add(a.im, b.re);
      q.add(a.re, b.im);
    } else {
      p.add(a.re, b.re);
      q.add(a.im, b.im);
      s.add(a.re, b.im);
      s.add(a.im, b.re);
    }
  }
  QCD_HD int64_t re() const { return CONJ ? s.value() : fx_diff(p, q); }
  QCD_HD int64_t im() const { return CONJ ? fx_diff(p, q) : s.value(); }
  QCD_HD FxC limbs(uint32_t& bad) const {
    const int64_t r = re(), i = im();
    fx_check(r, bad);
    fx_check(i, bad);
    return {fx_limbs(r), fx_limbs(i)};
  }
};

template <bool CONJ>
QCD_HD FxC fx_mul(const FxC& a, const FxC& b, uint32_t& bad) {
  FxDot<CONJ> d;
  d.add(a, b);
  return d.limbs(bad);
}

QCD_HD int fx_clz(uint64_t v) {
#ifdef __CUDA_ARCH__
  return __clzll(int64_t(v));
#else
  return v ? __builtin_clzll(v) : 64;
#endif
}
QCD_HD uint64_t fx_abs(int64_t v) { return v < 0 ? 0 - uint64_t(v) : uint64_t(v); }
// At least the largest |w_k|, below its next power of two.
QCD_HD uint64_t fx_size4(const int64_t w[4]) { return fx_abs(w[0]) | fx_abs(w[1]) | fx_abs(w[2]) | fx_abs(w[3]); }

// Whether every part of a staple sum of SU(2) links is below 2^-5 (relative errors
// would pass 2^-50): two in 10^7 random sums of six unit quaternions.
QCD_HD bool fx_small(const int64_t A[4]) { return (fx_size4(A) >> (FX_UNIT - 5)) == 0; }
// The same for a subgroup block of U A / 8 (twice the block), U or A small: all below
// 2^-8, one in 10^7 blocks of random links.
QCD_HD bool fx_small_block(const int64_t w[4]) { return (fx_size4(w) >> (FX_UNIT - 8)) == 0; }
// Collects the parts of a row or a quaternion; fx_tiny: all were below 1/4, which a unit
// one's are not (1/2 of the largest of four, 0.4 of six).
QCD_HD uint32_t fx_part(Fx v) { return uint32_t(v.hi ^ (v.hi >> 31)); }
QCD_HD bool fx_tiny(uint32_t parts) { return (parts >> (FX_LIMB - 2)) == 0; }

// 1 / n for n in [1/4, 4) (2^58 units): a 24-bit seed y = 2^-27 yi (absolute
// error below 2^-23 of it) and one step of third order, y (1 + e + e^2) with
// e = 1 - n y formed exactly to 2^-58.  At most 4 - 2^-58, the largest number that
// two limbs hold: n = 1/4 is met exactly (one component of a normalised block), and
// rounded down n may read a few units less where the norm is not below 1/4.
QCD_HD int64_t fx_reciprocal(int64_t n) {
  const Fx l = fx_limbs(n);
  const float f = float(l.hi > 0 ? l.hi : 1);  // n 2^29
#ifdef __CUDA_ARCH__
  const int32_t yi = __float2int_rn(__fdividef(72057594037927936.f, f));  // 2^56 / f = y 2^27
#else
  const int32_t yi = int32_t(72057594037927936.f / f + 0.5f);
#endif
  const int64_t prod = fx_add(fx_mad(l.hi, yi, 0) << 2, fx_mad(l.lo, yi, 0) >> 27);
  const int64_t e = fx_sub(int64_t(1) << FX_UNIT, prod);
  const int32_t es = int32_t(e >> 18);
  const int64_t t = e + (fx_mad(es, es, 0) >> 22);
  const int64_t y = (int64_t(yi) << 31) + ((int64_t(yi) * (t >> 2)) >> 25);
  constexpr int64_t top = (int64_t(1) << (FX_UNIT + 2)) - 1;
  return y < top ? y : top;
}

// Left-normalises the quaternion w so that its largest component is in
// [1/2, 1); returns 0 for w = 0.
QCD_HD bool fx_normalise4(int64_t w[4]) {
  const uint64_t m = fx_size4(w);
  if (m == 0) return false;
  const int z = fx_clz(m) - 1;
  for (int k = 0; k < 4; ++k) w[k] = int64_t(uint64_t(w[k]) << z) >> 5;
  return true;
}

// The overrelaxation rotation of a subgroup block w (any scale): r = (v^+)^2
// with v = w / |w|, i.e. r0 = 2 w0^2 / |w|^2 - 1, r_k = -2 w0 w_k / |w|^2.
// False for w = 0.
QCD_HD bool fx_overrelax(int64_t w[4], Fx r[4]) {
  if (!fx_normalise4(w)) return false;
  Fx l[4];
  FxAcc n;
  for (int k = 0; k < 4; ++k) {
    l[k] = fx_limbs(w[k]);
    n.add(l[k], l[k]);
  }
  FxAcc s;
  s.add(l[0], fx_limbs(fx_reciprocal(n.value())));
  const Fx sl = fx_limbs(s.value());  // w0 / |w|^2, at most 2
  for (int k = 0; k < 4; ++k) {
    FxAcc t;
    t.add(l[k], sl);
    const int64_t v = t.value() * 2;
    r[k] = fx_limbs(k == 0 ? v - (int64_t(1) << FX_UNIT) : -v);
  }
  return true;
}

// u <- V^+ u^+ V^+ = 2 <V^+, u> V^+ - u for the unit quaternion V = A / |A| (A of any
// scale): the overrelaxation of an SU(2) link.  False, and u as it was, for A = 0.
// u is read with components below 2; what a link off the group can take out of range
// (the product with the normalised block reaches 2 |u|, the result |u|) is checked
// before it is cut into limbs.
QCD_HD bool fx_reflect(int64_t A[4], Fx u[4], uint32_t& bad) {
  if (!fx_normalise4(A)) return false;
  Fx w[4];
  FxAcc n, d;
  for (int k = 0; k < 4; ++k) {
    w[k] = fx_limbs(k ? -A[k] : A[k]);
    n.add(w[k], w[k]);
    d.add(w[k], u[k]);
  }
  const int64_t dv = d.value();
  fx_check(dv, bad);
  FxAcc f;
  f.add(fx_limbs(dv), fx_limbs(fx_reciprocal(n.value())));
  const int64_t fv = f.value();  // at most |u| / |A| with A normalised above 1/2
  fx_check(fv, bad);
  const Fx s = fx_limbs(fv);
  for (int k = 0; k < 4; ++k) {
    FxAcc t;
    t.add(w[k], s);
    const int64_t v = fx_sub(2 * t.value(), fx_value(u[k]));
    fx_check(v, bad);
    u[k] = fx_limbs(v);
  }
  return true;
}

#ifdef __CUDACC__
// Sum of v (2^-58 units) over the warp, exact: three words of 22, 22 and 20 bits by
// the integer reduction instruction, then one rounding.
__device__ __forceinline__ double fx_warp_sum(int64_t v) {
  const unsigned lo = __reduce_add_sync(0xffffffffu, unsigned(v) & 0x3fffffu);
  const unsigned mid = __reduce_add_sync(0xffffffffu, unsigned(uint64_t(v) >> 22) & 0x3fffffu);
  const int hi = __reduce_add_sync(0xffffffffu, int(v >> 44));
  // hi 2^44 + mid 2^22 + lo in 2^-58 units: below 2^69, so the two upper words in FP64
  return double(hi) * 0x1p-14 + double((int64_t(mid) << 22) + int64_t(lo)) * 0x1p-58;
}
#endif

QCD_HD Fx fx_neg(Fx a) { return {-a.hi, -a.lo}; }
QCD_HD FxC fx_conj(FxC a) { return {a.re, fx_neg(a.im)}; }

// v + v d for a small d
QCD_HD Fx fx_scale1p(Fx v, Fx d) {
  FxAcc s;
  s.add(v, d);
  return fx_limbs(fx_add(fx_value(v), s.value()));
}

// 1/sqrt(n) - 1 for a squared norm n within 2^-19 of 1: -e/2 + 3 e^2/8 to below
// 2^-58.  False when it is further off.
QCD_HD bool fx_unit_factor(int64_t n, Fx& d) {
  const int64_t e = fx_sub(n, int64_t(1) << FX_UNIT);
  if (fx_abs(e) >> 39) return false;
  const int32_t es = int32_t(e >> 8);
  d = fx_limbs(-(e >> 1) + ((3 * (fx_mad(es, es, 0) >> 3)) >> 42));
  return true;
}

QCD_HD bool fx_unit3(FxC v[3]) {
  FxAcc n;
  for (int k = 0; k < 3; ++k) {
    n.add(v[k].re, v[k].re);
    n.add(v[k].im, v[k].im);
  }
  Fx d;
  if (!fx_unit_factor(n.value(), d)) return false;
  for (int k = 0; k < 3; ++k) v[k] = {fx_scale1p(v[k].re, d), fx_scale1p(v[k].im, d)};
  return true;
}

// Gram-Schmidt of rows 0 and 1 of a near-unitary matrix and row 2 =
// conj(row 0 x row 1).  False when the rows are too far from it.
QCD_HD bool fx_reunit(FxC m[3][3]) {
  uint32_t bad = 0;
  if (!fx_unit3(m[0])) return false;
  FxDot<true> p;
  for (int k = 0; k < 3; ++k) p.add(m[1][k], m[0][k]);
  const FxC c = p.limbs(bad);
  for (int k = 0; k < 3; ++k) {
    FxDot<false> d;
    d.add(c, m[0][k]);
    m[1][k] = {fx_limbs(fx_sub(fx_value(m[1][k].re), d.re())), fx_limbs(fx_sub(fx_value(m[1][k].im), d.im()))};
  }
  if (!fx_unit3(m[1])) return false;
  for (int k = 0; k < 3; ++k) {
    const int k1 = (k + 1) % 3, k2 = (k + 2) % 3;
    const FxC b = m[0][k2], nb{fx_neg(b.re), fx_neg(b.im)};
    FxDot<false> d;
    d.add(m[0][k1], m[1][k2]);
    d.add(nb, m[1][k1]);
    m[2][k] = fx_conj(d.limbs(bad));
  }
  return !(bad & FX_BAD);
}

}  // namespace qcd
