"""The sums of FP32 terms (qcd_sums.cuh) run by the host compiler: as close to the exact
sum as FP64 can say (two roundings of it), for a thread's and a warp's worth of terms
and for thousands of them (two numbers: for one term a lane); infinities and NaN as an FP64 sum gives them."""
import os
import subprocess

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1310_7087_gb300", "csrc")

PROGRAM = r"""
#include "qcd_sums.cuh"
#include <cstdio>
#include <initializer_list>
#include <random>
using qcd::SumF;
double worst = 0;
template <class Sum>
void sums(std::initializer_list<int> counts) {
  std::mt19937_64 g(1);
  std::uniform_real_distribution<float> u(0.f, 3.f);
  for (int n : counts)
    for (int it = 0; it < (n > 100 ? 20 : 2000); ++it) {
      Sum lane[32];
      __int128 exact = 0, size = 0;  // units of 2^-40: the terms are multiples of it
      for (int l = 0; l < 32; ++l)
        for (int k = 0; k < n; ++k) {
          float v = std::nearbyint(u(g) * 0x1p20f) * 0x1p-20f + std::nearbyint(u(g) * 0x1p19f) * 0x1p-40f;
          if (it & 1 && k & 1) v = -v;
          lane[l].add(v);
          const long long w = (long long)(double(v) * 0x1p40);
          exact += w;
          size += w < 0 ? -w : w;
        }
      for (int off = 16; off; off >>= 1)
        for (int l = 0; l < off; ++l) lane[l].merge(lane[l + off]);
      const __int128 got = (__int128)(lane[0].value() * 0x1p60), d = got - (exact << 20);
      const double err = double(d < 0 ? -d : d) / double(size << 20);
      if (err > worst) worst = err;
    }
}
int main() {
  sums<SumF>({1, 3, 6, 40, 1000, 20000});
  sums<qcd::SumF32>({1});
  SumF a, b, c, d;
  const float inf = HUGE_VALF;
  for (float v : {1.f, inf, 2.f}) a.add(v);
  for (float v : {1.f, -inf, inf}) b.add(v);
  for (float v : {1.f, NAN, inf}) c.add(v);
  d.add(-inf);
  SumF e, f = a;
  e.add(2.f);
  e.merge(d);
  f.merge(d);
  const int ok = a.value() == HUGE_VAL && b.value() != b.value() && c.value() != c.value() && e.value() == -HUGE_VAL &&
                 f.value() != f.value();
  printf("%g %d\n", worst, ok);
}
"""


def test_fp32_sums(tmp_path):
    src, exe = tmp_path / "sums.cpp", tmp_path / "sums"
    src.write_text(PROGRAM)
    subprocess.run(["g++", "-O2", "-I" + CSRC, "-x", "c++", str(src), "-o", str(exe)], check=True)
    out = subprocess.run([str(exe)], check=True, capture_output=True, text=True).stdout.split()
    assert float(out[0]) < 2.0 ** -52 and out[1] == "1", out
