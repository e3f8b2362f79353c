// dfloat.cuh -- FP32 pairs (hi + lo) that stand for values of about 48 significant
// bits, with the error bounds of df.cu: the double-float pass and the rows of folded
// nets (prologue.cu) are computed in them, on a part that runs FP64 at a
// sixty-fourth of its FP32 rate.
#pragma once
#include <cuda_runtime.h>

namespace vbmc {

__device__ __forceinline__ float2 two_sum(float a, float b) {
    const float s = __fadd_rn(a, b);
    const float bb = __fsub_rn(s, a);
    const float e = __fadd_rn(__fsub_rn(a, __fsub_rn(s, bb)), __fsub_rn(b, bb));
    return make_float2(s, e);
}

__device__ __forceinline__ float2 df_add(float2 a, float2 b) {
    const float2 s = two_sum(a.x, b.x);
    return two_sum(s.x, __fadd_rn(s.y, __fadd_rn(a.y, b.y)));
}

// an FP64 value as a pair: |v - (hi + lo)| <= 2^-48 |v|
__device__ __forceinline__ float2 split64(double v) {
    const float hi = (float)v;
    return make_float2(hi, (float)(v - (double)hi));
}

__device__ __forceinline__ float abs_up(float2 a) { return __fmul_ru(fabsf(a.x), 1.f + 0x1p-22f); }

}  // namespace vbmc
