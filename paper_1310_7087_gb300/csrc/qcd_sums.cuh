// qcd_sums.cuh -- sums of FP32 terms without FP64 arithmetic.
//
// One FP64 add of a warp takes 64 cycles of an SM sub-partition, and so does a
// conversion, so FP32 terms are summed by Knuth's error-free TwoSum (t + e = s + v
// exactly), the errors by a second one, and the sum is formed in FP64 once per warp.
// What is lost is the rounding of the second errors, 2^-72 of the sum and step: less
// than FP64 sums lose for any number of terms that a thread meets.  Plain C++, so that
// the host compiler can run the same arithmetic.
#pragma once

#include "qcd_fix.cuh"  // QCD_HD

namespace qcd {

// K = 3 as above.  K = 2, the errors in one rounded number: for one term a lane, 32 in
// all, whose errors it still holds (3e-15 of the sum lost at 6 terms a lane, 2e-13 at
// 20,000); a third number costs the last pass of SU(3) 48^3x16 3 us a phase of 95.
template <int K>
struct FloatSum {
  float s = 0.f, c = 0.f, cc = 0.f;
  // s <- s + v, returns what was rounded off
  QCD_HD static float two_sum(float& s, float v) {
    const float t = s + v, b = t - s, e = (s - (t - b)) + (v - b);
    s = t;
    return e;
  }
  QCD_HD void add(float v) {
    const float e = two_sum(s, v);
    if (K == 3) cc += two_sum(c, e);
    else c += e;
  }
  QCD_HD void merge(const FloatSum& o) {
    const float e = two_sum(s, o.s);
    if (K == 3) {
      const float f = two_sum(c, o.c);
      cc += o.cc + (f + two_sum(c, e));
    } else {
      c += o.c + e;
    }
  }
  // (an infinite sum's errors are NaN)
  QCD_HD double value() const { return s - s == 0.f ? double(s) + (double(c) + double(cc)) : double(s); }
#ifdef __CUDACC__
  __device__ __forceinline__ void merge_down(int off) {
    FloatSum o;
    o.s = __shfl_down_sync(0xffffffffu, s, off);
    o.c = __shfl_down_sync(0xffffffffu, c, off);
    if (K == 3) o.cc = __shfl_down_sync(0xffffffffu, cc, off);
    merge(o);
  }
#endif
};
using SumF = FloatSum<3>;
using SumF32 = FloatSum<2>;

#ifdef __CUDACC__
// value() of N sums that lane 0 of a warp holds, sum k in lane 3 k: each of the 3 N
// numbers converted by a lane of its own, so that the warp takes one conversion and
// two FP64 adds (five of these instructions for each sum in lane 0 made working sweeps
// of SU(2) 32^3x8 135 us instead of 127).
template <int K, int N>
__device__ __forceinline__ double warp_values(const FloatSum<K> (&v)[N]) {
  const int lane = threadIdx.x & 31;
  float x = 0.f;
#pragma unroll
  for (int k = 0; k < N; ++k) {
    const float s = __shfl_sync(0xffffffffu, v[k].s, 0), c = __shfl_sync(0xffffffffu, v[k].c, 0),
                cc = K == 3 ? __shfl_sync(0xffffffffu, v[k].cc, 0) : 0.f;
    if (lane == 3 * k) x = s;
    if (lane == 3 * k + 1) x = c;
    if (lane == 3 * k + 2) x = cc;
  }
  const double d = x, e = K == 3 ? d + __shfl_down_sync(0xffffffffu, d, 1) : d;
  const double r = d + __shfl_down_sync(0xffffffffu, e, 1);
  return x - x == 0.f ? r : d;
}
#endif

}  // namespace qcd
