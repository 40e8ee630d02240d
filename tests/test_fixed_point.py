"""The fixed-point arithmetic of the FP64 kernels (qcd_fix.cuh, qcd_fixmath.cuh)
run by the host compiler against long double: every function within 2^-54, half
the spacing of FP64 numbers in [1/2, 1) (the arithmetic works in 2^-58 units;
its longest chain sums about ten truncations); the heat-bath draw's exponent no
further off than the same expression in double."""
import os
import platform
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1310_7087_gb300", "csrc")

PROGRAM = r"""
#include "qcd_fixmath.cuh"
#include <cstdio>
#include <random>
using namespace qcd;
typedef long double L;
static const L U = (L)(1ll << 58), PI = 3.14159265358979323846264338327950288L;
int main() {
  std::mt19937_64 g(1);
  std::uniform_real_distribution<double> u(-1, 1);
  L dot = 0, rec = 0, orr = 0, lg = 0, trig = 0, rs = 0, sq = 0, kp = 0, kpd = 0, dir = 0, re = 0;
  int flags = 0;
  for (long it = 0; it < 400000; ++it) {
    double a[6], b[6];
    L na = 0, nb = 0, s = 0;
    for (int k = 0; k < 6; ++k) { a[k] = u(g); b[k] = u(g); na += a[k] * a[k]; nb += b[k] * b[k]; }
    for (int k = 0; k < 6; ++k) { a[k] /= sqrtl(na); b[k] /= sqrtl(nb); }
    uint32_t big = 0, bad = 0;
    FxDot<true> d;
    for (int k = 0; k < 3; ++k) {
      const FxC x{fx_load(a[2 * k], big), fx_load_int(a[2 * k + 1], big)};
      const FxC y{fx_load_int(b[2 * k], big), fx_load(b[2 * k + 1], big)};
      d.add(x, y);
      s += (L)a[2 * k] * b[2 * k] + (L)a[2 * k + 1] * b[2 * k + 1];
    }
    d.limbs(bad);
    flags += (big & FX_BIG) || (bad & FX_BAD);
    dot = fmaxl(dot, fabsl(d.re() / U - s));
    const int64_t n = (int64_t)((0.25L + 3.7499999L * (0.5L + 0.5L * u(g))) * U);
    rec = fmaxl(rec, fabsl(fx_reciprocal(n) / U * (n / U) - 1));
    rs = fmaxl(rs, fabsl(fx_rsqrt(n) / U * sqrtl(n / U) - 1));
    const int64_t y = (int64_t)(g() >> (6 + it % 40));
    sq = fmaxl(sq, fabsl(fx_sqrt(y) / U - sqrtl(y / U)));
    int64_t w[4];
    L v[4], n2 = 0;
    for (int k = 0; k < 4; ++k) { w[k] = (int64_t)(u(g) * ldexpl(3.9L, -(int)(it % 12)) * U); v[k] = w[k] / U; n2 += v[k] * v[k]; }
    Fx r[4];
    // (a component of 2^-12 carries 46 bits, so its rotation is compared at full size only)
    if (it % 12 == 0 && fx_overrelax(w, r))
      for (int k = 0; k < 4; ++k) orr = fmaxl(orr, fabsl(fx_value(r[k]) / U - (k ? -2 * v[0] * v[k] / n2 : 2 * v[0] * v[0] / n2 - 1)));
    uint32_t w0 = g(), w1 = g(), w2 = g();
    if (it % 5 == 0) w0 |= 0xffffff00u << (it % 7);
    if (it % 13 == 0) w0 = (it % 512) << 9;
    int z; int64_t e, c, sn;
    const uint32_t o = fx_odd24(w0);
    fx_neglog24(o, z, e);
    lg = fmaxl(lg, fabsl(((L)z * FX_LN2 + e) / U + logl(ldexpl(o, -24))) / fmaxl(1, z));
    fx_sincos(o << 8, c, sn);
    const L an = 2 * PI * ldexpl((L)(uint32_t)(o << 8), -32);
    trig = fmaxl(trig, fmaxl(fabsl(c / U - cosl(an)), fabsl(sn / U - sinl(an))));
    const L u0 = ldexpl(o, -24), u1 = ldexpl(fx_odd24(w1), -24), u2 = ldexpl(fx_odd24(w2), -24), cc = cosl(2 * PI * u2);
    const L ex = -logl(u1) - logl(u0) * cc * cc;
    // of a value up to 33, whose cosine's error is multiplied by -ln u1: against the same expression in double
    const double d2 = cos(2 * M_PI * (double)u2);
    kp = fmaxl(kp, fabsl(2 * fx_kp_e(w0, w1, w2) / U - ex));
    kpd = fmaxl(kpd, fabsl(-log((double)u1) - log((double)u0) * d2 * d2 - ex));
    int64_t t[3];
    fx_direction(w0, w1, t);
    const L st = 2 * sqrtl(u0 * (1 - u0));
    dir = fmaxl(dir, fmaxl(fabsl(t[0] / U - st * cosl(2 * PI * u1)), fmaxl(fabsl(t[1] / U - st * sinl(2 * PI * u1)), fabsl(t[2] / U - (2 * u0 - 1)))));
    // rows next to unitary: unit rows, orthogonal, to the last bits
    FxC m[3][3];
    L q[6], dt = 0, di = 0;
    for (int k = 0; k < 3; ++k) { dt += (L)a[2 * k] * b[2 * k] + (L)a[2 * k + 1] * b[2 * k + 1]; di += (L)a[2 * k] * b[2 * k + 1] - (L)a[2 * k + 1] * b[2 * k]; }
    L nq = 0;
    for (int k = 0; k < 3; ++k) { q[2 * k] = b[2 * k] - (dt * a[2 * k] - di * a[2 * k + 1]); q[2 * k + 1] = b[2 * k + 1] - (dt * a[2 * k + 1] + di * a[2 * k]); nq += q[2 * k] * q[2 * k] + q[2 * k + 1] * q[2 * k + 1]; }
    for (int k = 0; k < 3; ++k) {
      m[0][k] = {fx_load(a[2 * k] * (1 + 1e-7), big), fx_load(a[2 * k + 1] * (1 + 1e-7), big)};
      m[1][k] = {fx_load((double)(q[2 * k] / sqrtl(nq)) + 1e-7 * a[2 * k], big), fx_load((double)(q[2 * k + 1] / sqrtl(nq)), big)};
    }
    if (!fx_reunit(m)) { ++flags; continue; }
    for (int i = 0; i < 3; ++i) for (int j = 0; j <= i; ++j) {
      L x = 0, y2 = 0;
      for (int k = 0; k < 3; ++k) {
        const L ar = fx_value(m[i][k].re) / U, ai = fx_value(m[i][k].im) / U, br = fx_value(m[j][k].re) / U, bi = fx_value(m[j][k].im) / U;
        x += ar * br + ai * bi; y2 += ai * br - ar * bi;
      }
      re = fmaxl(re, fmaxl(fabsl(x - (i == j)), fabsl(y2)));
    }
  }
  // what is out of range is reported
  uint32_t b1 = 0, b2 = 0, b3 = 0, b4 = 0;
  fx_load(2.0, b1); fx_load(-1e300, b2); fx_load_int(HUGE_VAL, b3); fx_load_int(NAN, b4);
  uint32_t c1 = 0, c2 = 0, c3 = 0;
  fx_check(int64_t(1) << 59, c1); fx_check(-(int64_t(1) << 59) - 1, c2); fx_check((int64_t(1) << 59) - 1, c3); fx_check(-(int64_t(1) << 59), c3);
  const int ok = (b1 & b2 & b3 & b4 & FX_BIG) && (c1 & FX_BAD) && (c2 & FX_BAD) && !(c3 & FX_BAD);
  printf("%Lg %Lg %Lg %Lg %Lg %Lg %Lg %Lg %Lg %Lg %d %d\n", dot, rec, orr, lg, trig, rs, sq, kp / kpd * ldexpl(1, -54), dir, re, flags, ok);
}
"""


@pytest.mark.skipif(platform.machine() not in ("x86_64", "aarch64"), reason="needs a long double wider than double")
def test_fixed_point_functions(tmp_path):
    src, exe = tmp_path / "fix.cpp", tmp_path / "fix"
    src.write_text(PROGRAM)
    subprocess.run(["g++", "-O2", "-I" + CSRC, "-x", "c++", str(src), "-o", str(exe)], check=True)
    out = subprocess.run([str(exe)], check=True, capture_output=True, text=True).stdout.split()
    names = ("dot product", "reciprocal", "overrelaxation", "logarithm", "circle", "1/sqrt", "sqrt", "draw", "direction",
             "unitarity")
    for name, err in zip(names, out):
        # the rotation squares a unit vector: twice its error; so does u u^+
        bound = 2.0 ** (-53 if name in ("overrelaxation", "unitarity") else -54)
        assert float(err) < bound, (name, err)
    assert out[-2:] == ["0", "1"], out
