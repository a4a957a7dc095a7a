// float_sums.cuh -- sums kept in three floats, on the FP32 pipes (the FP64 pipe
// does two operations per cycle and SM): 2^-64 of the sum of magnitudes for some
// hundred terms, below the rounding of a sum in double.  (The _rn intrinsics keep
// the rounded steps from being contracted into fused multiply-adds, which would
// break the error-free transformations.)
#pragma once

namespace ace {

// s += x (TwoSum); returns the error.
__device__ __forceinline__ float two_sum(float& s, float x) {
    const float t = __fadd_rn(s, x), b = __fsub_rn(t, s);
    const float e = __fadd_rn(__fsub_rn(s, __fsub_rn(t, b)), __fsub_rn(x, b));
    s = t;
    return e;
}
// (s, e, ee) += x: TwoSum's error goes to e by a TwoSum of its own, whose error is
// added up in ee (A. Klein, A generalized Kahan-Babuska-summation algorithm,
// Computing 76 (2006)).
__device__ __forceinline__ void sum_add3(float& s, float& e, float& ee, float x) {
    ee = __fadd_rn(ee, two_sum(e, two_sum(s, x)));
}
__device__ __forceinline__ void sum_merge3(float& s, float& e, float& ee, float s2, float e2, float ee2) {
    sum_add3(s, e, ee, s2);
    ee = __fadd_rn(ee, __fadd_rn(two_sum(e, e2), ee2));
}

}  // namespace ace
