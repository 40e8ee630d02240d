"""The fixed-point arithmetic of the FP64 kernels (qcd_fix.cuh, qcd_fixmath.cuh) at
the ends of its ranges, run by the host compiler against long double.  Bounds: a
few units of 2^-58 per function, as in test_fixed_point (2^-54, and 2^-53 where a
unit vector is squared)."""
import os
import platform
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1310_7087_gb300", "csrc")

pytestmark = pytest.mark.skipif(platform.machine() not in ("x86_64", "aarch64"),
                                reason="needs a long double wider than double")

HEAD = r"""
#include "qcd_fixmath.cuh"
#include <cstdio>
#include <random>
using namespace qcd;
typedef long double L;
static const L U = (L)(1ll << 58), PI = 3.14159265358979323846264338327950288L;
// the 24 units of the Hurwitz quaternions (the first 8: the quaternion group)
static void hurwitz(int i, double q[4]) {
  for (int k = 0; k < 4; ++k) q[k] = i < 8 ? (i >> 1) == k ? 1 - 2 * (i & 1) : 0.0 : 0.5 - ((i - 8) >> k & 1);
}
static int64_t units(double x) { return (int64_t)(x * (double)(1ll << 58)); }
static Fx limbs(double x) { uint32_t b = 0; return fx_load(x, b); }
"""


def run(tmp_path, body):
    src, exe = tmp_path / "fix.cpp", tmp_path / "fix"
    src.write_text(HEAD + body)
    subprocess.run(["g++", "-O2", "-I" + CSRC, "-x", "c++", str(src), "-o", str(exe)], check=True)
    return subprocess.run([str(exe)], check=True, capture_output=True, text=True).stdout.split()


def test_reciprocal_ends(tmp_path):
    """1/n next to 1/4 and to 4, through the limbs that its users cut it into.  The
    squared norm of a normalised block may read a few units below 1/4 (products
    are rounded down) while the norm is not below it: 1/n is then within 2^-52 of 4."""
    out = run(tmp_path, r"""
int main() {
  L err = 0, below = 0;
  for (int64_t d = -16; d < 200000; ++d) {
    for (int end = 0; end < 2; ++end) {
      const int64_t n = end ? (int64_t(1) << 60) - 17 - d : (int64_t(1) << 56) + d;
      const L y = fx_value(fx_limbs(fx_reciprocal(n))) / U;
      if (!end && d < 0) below = fmaxl(below, fabsl(y - 4));
      else err = fmaxl(err, fabsl(y * (n / U) - 1));
    }
  }
  printf("%Lg %Lg\n", err, below);
}
""")
    assert float(out[0]) < 2.0 ** -54 and float(out[1]) < 2.0 ** -52, out


def test_overrelaxation_of_exact_blocks(tmp_path):
    """The SU(3) subgroup rotation and the SU(2) reflection for staples that are a
    multiple of a Hurwitz quaternion (cold links with centre elements among them) and
    for a block with one large component."""
    out = run(tmp_path, r"""
int main() {
  L rot = 0, refl = 0;
  int bad_links = 0;
  std::mt19937_64 g(1);
  std::normal_distribution<double> z;
  auto check = [&](const int64_t A[4]) {
    L v[4], n2 = 0;
    for (int k = 0; k < 4; ++k) { v[k] = A[k] / U; n2 += v[k] * v[k]; }
    int64_t w[4] = {A[0], A[1], A[2], A[3]};
    Fx r[4];
    fx_overrelax(w, r);
    for (int k = 0; k < 4; ++k)
      rot = fmaxl(rot, fabsl(fx_value(r[k]) / U - (k ? -2 * v[0] * v[k] / n2 : 2 * v[0] * v[0] / n2 - 1)));
    for (int i = 0; i < 40; ++i) {
      double q[4], m = 0;
      if (i < 24) hurwitz(i, q);
      else {
        for (int k = 0; k < 4; ++k) { q[k] = z(g); m += q[k] * q[k]; }
        for (int k = 0; k < 4; ++k) q[k] /= sqrt(m);
      }
      Fx u[4];
      L dot = 0;
      for (int k = 0; k < 4; ++k) { u[k] = limbs(q[k]); w[k] = A[k]; dot += (k ? -v[k] : v[k]) * (fx_value(u[k]) / U); }
      uint32_t bad = 0;
      fx_reflect(w, u, bad);
      if (bad & FX_BAD) { ++bad_links; continue; }
      L e[4];
      for (int k = 0; k < 4; ++k) e[k] = 2 * dot / n2 * (k ? -v[k] : v[k]) - (L)q[k];
      for (int k = 0; k < 4; ++k) refl = fmaxl(refl, fabsl(fx_value(u[k]) / U - e[k]));
    }
  };
  for (int i = 0; i < 24; ++i)
    for (double s : {1.0, 2.0, 3.0, 4.0, 5.0, 6.0, 0.5, 0.25}) {
      double q[4];
      hurwitz(i, q);
      const int64_t A[4] = {units(s * q[0]), units(s * q[1]), units(s * q[2]), units(s * q[3])};
      check(A);
    }
  for (int p = 54; p < 61; ++p)
    for (int m = 0; m < 32; ++m) {
      int64_t A[4];
      for (int k = 0; k < 4; ++k) A[k] = m >> k & 1 ? -1 : 0;
      A[m & 3] = m & 16 ? -(int64_t(1) << p) : int64_t(1) << p;
      check(A);
    }
  printf("%Lg %Lg %d\n", rot, refl, bad_links);
}
""")
    assert float(out[0]) < 2.0 ** -53 and float(out[1]) < 2.0 ** -53 and out[2] == "0", out


def test_rsqrt_ends(tmp_path):
    """1/sqrt(n) next to 1/4 (where a rounded seed can reach 2, and rounded down n may
    read a few units less) and to 4."""
    out = run(tmp_path, r"""
int main() {
  L err = 0;
  auto check = [&](int64_t n) { err = fmaxl(err, fabsl(fx_rsqrt(n) / U * sqrtl(n / U) - 1)); };
  for (int64_t d = 0; d < 200000; ++d) { check((int64_t(1) << 56) + d); check((int64_t(1) << 60) - 1 - d); }
  for (int64_t d = 1; d <= 16; ++d) check((int64_t(1) << 56) - d);
  for (int p = 17; p < 36; ++p)
    for (int64_t d = 0; d < 20000; ++d) check((int64_t(1) << 56) + (d << p) / 7);
  printf("%Lg\n", err);
}
""")
    assert float(out[0]) < 2.0 ** -54, out


def test_reflection_of_links_off_the_group(tmp_path):
    """Links whose components are below 2 but whose norm reaches 4: reflected to within
    four times a unit link's bound, or reported as out of range."""
    out = run(tmp_path, r"""
int main() {
  std::mt19937_64 g(2);
  std::normal_distribution<double> z;
  std::uniform_real_distribution<double> un(0.3, 4.0);
  L err = 0;
  long fixed = 0, unit_bad = 0;
  for (long it = 0; it < 2000000; ++it) {
    double a[4], q[4], na = 0, nq = 0;
    for (int k = 0; k < 4; ++k) { a[k] = z(g); q[k] = z(g); na += a[k] * a[k]; nq += q[k] * q[k]; }
    const double ra = un(g) * 1.5 / sqrt(na), rq = (it % 4 ? un(g) : 1.0) / sqrt(nq);
    bool inside = true;
    if (it % 3 == 0)  // a link along the staple's adjoint: the largest product
      for (int k = 0; k < 4; ++k) q[k] = (k ? -1 : 1) * a[k] / sqrt(na) * sqrt(nq) + 0.05 * q[k];
    Fx u[4];
    int64_t w[4];
    L v[4], n2 = 0, dot = 0;
    for (int k = 0; k < 4; ++k) {
      inside &= fabs(q[k] * rq) < 2;
      w[k] = units(a[k] * ra); v[k] = w[k] / U; n2 += v[k] * v[k];
    }
    if (!inside) continue;
    for (int k = 0; k < 4; ++k) { u[k] = limbs(q[k] * rq); dot += (k ? -v[k] : v[k]) * (fx_value(u[k]) / U); }
    L e[4];
    for (int k = 0; k < 4; ++k) e[k] = 2 * dot / n2 * (k ? -v[k] : v[k]) - fx_value(u[k]) / U;
    uint32_t bad = 0;
    fx_reflect(w, u, bad);
    if (bad & FX_BAD) { unit_bad += it % 4 == 0 && it % 3; continue; }
    ++fixed;
    for (int k = 0; k < 4; ++k) err = fmaxl(err, fabsl(fx_value(u[k]) / U - e[k]));
  }
  printf("%Lg %ld %ld\n", err, fixed, unit_bad);
}
""")
    assert float(out[0]) < 2.0 ** -51 and int(out[1]) > 500000 and out[2] == "0", out


def test_drawn_quaternion(tmp_path):
    """X = (1 - delta, sqrt(delta (2 - delta)) n) of the Kennedy-Pendleton draw at couplings from strong to weak:
    no further from long double than the same expressions in double, in the largest error and in the mean square.
    Every eighth draw has an exponent next to 0, where the modulus magnifies its error (the smallest go to FP64)."""
    out = run(tmp_path, r"""
int main() {
  std::mt19937_64 g(3);
  long small = 0;
  for (double alpha : {3.0, 10.0, 100.0, 1e3, 1e4, 1e6}) {
    L fm = 0, dm = 0, f2 = 0, d2 = 0;
    for (long it = 0; it < 400000; ++it) {
      uint32_t w0 = g(), w1 = g(), w2 = g(), v0 = g(), v1 = g();
      if (it % 8 == 0) { w1 |= 0xffffffffu << (9 + it / 8 % 16); w0 |= 0xffffffffu << (9 + it / 128 % 16); }
      const double u0 = ldexp(fx_odd24(w0), -24), u1 = ldexp(fx_odd24(w1), -24), u2 = ldexp(fx_odd24(w2), -24);
      const L c = cosl(2 * PI * u2), e = -logl(u1) - logl(u0) * c * c, delta = e / (L)alpha;
      if (delta >= 1.99L) continue;
      const double inv = 1.0 / alpha;
      const L p0 = ldexp(fx_odd24(v0), -24), ph = 2 * PI * ldexp(fx_odd24(v1), -24), st = 2 * sqrtl(p0 * (1 - p0)), r = sqrtl(delta * (2 - delta));
      const L X[4] = {1 - delta, r * st * cosl(ph), r * st * sinl(ph), r * (2 * p0 - 1)};
      // double
      const double cd = cos(2 * M_PI * u2), dd = (-log(u1) - log(u0) * cd * cd) * inv, q0 = (double)p0;
      const double sd = 2 * sqrt(q0 * (1 - q0)), rd = sqrt(dd * (2 - dd)), pd = 2 * M_PI * ldexp(fx_odd24(v1), -24);
      const double D[4] = {1 - dd, rd * sd * cos(pd), rd * sd * sin(pd), rd * (2 * q0 - 1)};
      // fixed point
      const double fe = double(fx_kp_e(w0, w1, w2));
      small += fx_kp_small(fe) && it % 8;
      if (fx_kp_small(fe)) continue;  // drawn in FP64
      const FxDelta fx(fe * inv);
      const int64_t fd = fx.value();
      int64_t n[3];
      fx_direction(v0, v1, n);
      const int64_t m = fx.modulus(fd);
      const int64_t F[4] = {FX_ONE - fd, fx_product(m, n[0]), fx_product(m, n[1]), fx_product(m, n[2])};
      L ef = 0, ed = 0;
      for (int k = 0; k < 4; ++k) { ef += (F[k] / U - X[k]) * (F[k] / U - X[k]); ed += (D[k] - X[k]) * (D[k] - X[k]); }
      fm = fmaxl(fm, ef); dm = fmaxl(dm, ed); f2 += ef; d2 += ed;
    }
    printf("%Lg %Lg ", sqrtl(fm / dm), sqrtl(f2 / d2));
  }
  // no try accepts delta >= 2
  int range = 1;
  for (double d : {0x1p58, 0x1.8p58, 0x1p63, 1e300, HUGE_VAL}) range &= FxDelta(d).value() >= 2 * FX_ONE;
  range &= FxDelta(0x1.fffffffffffffp57).value() < 2 * FX_ONE && FxDelta(0.0).value() == 0 && FxDelta(1e-300).value() == 0;
  printf("%ld\n", range ? small : -1);
}
""")
    assert len(out) == 13 and all(float(v) <= 1.0 for v in out[:-1]), out
    assert 0 <= int(out[-1]) < 5, out  # 2.1 million draws, one in 22 million expected
