// FP32 sums that keep their rounding errors.
#pragma once

namespace jerk {

// s + y: s becomes the rounded sum, the result is its exact error (Knuth's TwoSum)
__device__ __forceinline__ float two_sum(float &s, float y) {
    const float t = __fadd_rn(s, y);
    const float b = __fsub_rn(t, s);
    const float e = __fadd_rn(__fsub_rn(s, __fsub_rn(t, b)), __fsub_rn(y, b));
    s = t;
    return e;
}

}  // namespace jerk
