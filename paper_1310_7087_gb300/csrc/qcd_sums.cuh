// qcd_sums.cuh -- sums of FP32 terms without FP64 arithmetic.
//
// One FP64 add of a warp takes 64 cycles of an SM sub-partition, and so does a
// conversion, so FP32 terms are summed by Knuth's error-free TwoSum (t + e = s + v
// exactly), the errors by a second one, and the sum is formed in FP64 once per warp.
// What is lost is the rounding of the second errors, 2^-72 of the sum and step: less
// than FP64 sums lose for any number of terms that a thread meets.  (With the errors
// in one number, 4e-15 of the sum at 1,000 terms a thread, 2e-13 at 20,000.)  Plain
// C++, so that the host compiler can run the same arithmetic.
#pragma once

#include "qcd_fix.cuh"  // QCD_HD

namespace qcd {

struct SumF {
  float s = 0.f, c = 0.f, cc = 0.f;
  // s <- s + v, returns what was rounded off
  QCD_HD static float two_sum(float& s, float v) {
    const float t = s + v, b = t - s, e = (s - (t - b)) + (v - b);
    s = t;
    return e;
  }
  QCD_HD void add(float v) { cc += two_sum(c, two_sum(s, v)); }
  QCD_HD void merge(const SumF& o) {
    const float e = two_sum(s, o.s), f = two_sum(c, o.c);
    cc += o.cc + (f + two_sum(c, e));
  }
  // (an infinite sum's errors are NaN)
  QCD_HD double value() const { return s - s == 0.f ? double(s) + (double(c) + double(cc)) : double(s); }
#ifdef __CUDACC__
  __device__ __forceinline__ void merge_down(int off) {
    SumF o;
    o.s = __shfl_down_sync(0xffffffffu, s, off);
    o.c = __shfl_down_sync(0xffffffffu, c, off);
    o.cc = __shfl_down_sync(0xffffffffu, cc, off);
    merge(o);
  }
#endif
};

}  // namespace qcd
