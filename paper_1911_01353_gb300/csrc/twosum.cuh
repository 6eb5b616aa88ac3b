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

// The rounded sum of a partial's two lanes; what the rounding left (of a finite
// sum) stays as the next partial's start, so that one FP64 addition per partial
// loses nothing.
__device__ __forceinline__ float take_sum(float2 &v) {
    float t = v.x;
    const float e = two_sum(t, v.y);
    v = make_float2(fabsf(t) <= 3.402823466e38f ? e : 0.f, 0.f);
    return t;
}

}  // namespace jerk
