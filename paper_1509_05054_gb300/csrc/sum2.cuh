// A thread's sum of many FP32 values to more than FP32 precision.  Internal to the
// library.
#pragma once

namespace dlk {
namespace {

// The sum of non-negative values as an unevaluated FP32 pair (Knuth's two-sum: the
// rounding error of every addition goes to lo); FP64 additions run at 1/64 of the FP32
// rate.  Beside it the same sum in plain FP32, scaled by 2^-32, which stands in
// where the pair has passed the FP32 range, so that finite values sum to the finite
// FP64 value and an infinite or NaN one to itself.  (Moving the pair to FP64 when it
// grows large, a test and a branch per addition, cost k_small.cu 53 us of 333 and a
// proposer training pass 360 of 1,350; the scaled sum 6 and 4.)
struct Sum2 {
  float hi = 0.f, lo = 0.f, scaled = 0.f;
  __device__ __forceinline__ void add(float x) {
    const float s = __fadd_rn(hi, x), b = __fsub_rn(s, hi);
    lo = __fadd_rn(lo, __fadd_rn(__fsub_rn(hi, __fsub_rn(s, b)), __fsub_rn(x, b)));
    hi = s;
    scaled = __fmaf_rn(x, 0x1p-32f, scaled);
  }
  __device__ __forceinline__ double value() const {
    return isfinite(hi) ? (double)hi + (double)lo : (double)scaled * 0x1p32;
  }
};

}  // namespace
}  // namespace dlk
