// Products of float pairs (hi, lo: 48 significant bits of a float64) summed in
// compensated arithmetic on the FP32 units (error-free TwoProd and TwoSum,
// Ogita, Rump and Oishi 2005).
#pragma once
#include <cuda_runtime.h>

namespace svk {

// (s, c) += a b
__device__ __forceinline__ void dot2_add(float& s, float& c, float2 a, float2 b) {
    const float p = __fmul_rn(a.x, b.x);
    const float e = fmaf(a.x, b.x, -p);                      // a.hi b.hi = p + e exactly
    const float t = __fadd_rn(s, p), z = __fsub_rn(t, s);
    const float err = __fadd_rn(__fsub_rn(s, __fsub_rn(t, z)), __fsub_rn(p, z));  // s + p = t + err exactly
    s = t;
    c += err + e + fmaf(a.x, b.y, a.y * b.x);
}

__device__ __forceinline__ float2 pair_of(double d) {
    const float hi = (float)d;
    return make_float2(hi, (float)(d - (double)hi));
}

}  // namespace svk
