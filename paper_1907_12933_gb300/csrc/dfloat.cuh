// dfloat.cuh -- FP32 pairs (hi + lo) that stand for values of about 48 significant
// bits, with the error bounds of df.cu: the double-float pass, the rows of folded nets
// (prologue.cu) and the potentials of the covers over pairs (pairs.cu) are computed in
// them, on a part that runs FP64 at a sixty-fourth of its FP32 rate.
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

// Sum of products of FP32 numbers w and pairs h, as a pair. Settled after at most kSettle
// terms, n of them are off by at most (6.5 n + 20) 2^-48 S, S = sum of |w h|: with
// u = 2^-24 a step's part t.y + ep is below u S + 2 u |w h| and rounds by u times that, and
// a.y, below (1 + i) u S + 2 u |w h| summed over i terms since it was settled, rounds by
// u times that: 44 u^2 S for 8 terms, against n^2 / 2 u^2 S where it is never settled (17
// times the bound of 8 (n + 32) u^2 S at n = 1,024). Joining two sums (df_add) adds
// 3 u^2 of their magnitudes.
constexpr int kSettle = 8;

struct PairSum {
    float2 a = {0.f, 0.f};
    __device__ __forceinline__ void add(float w, float2 h) {
        const float pr = __fmul_rn(w, h.x);
        float ep = __fmaf_rn(w, h.x, -pr);
        ep = __fmaf_rn(w, h.y, ep);
        const float2 t = two_sum(a.x, pr);
        a = make_float2(t.x, __fadd_rn(a.y, __fadd_rn(t.y, ep)));
    }
    __device__ __forceinline__ void settle() { a = two_sum(a.x, a.y); }
};

// Two FP32 lanes in one 64-bit register (fma.rn.f32x2: two results an instruction).
typedef unsigned long long f32x2;

__device__ __forceinline__ f32x2 pack2(float a, float b) {
    f32x2 d;
    asm("mov.b64 %0, {%1, %2};" : "=l"(d) : "f"(a), "f"(b));
    return d;
}

__device__ __forceinline__ float2 unpack2(f32x2 v) {
    float2 d;
    asm("mov.b64 {%0, %1}, %2;" : "=f"(d.x), "=f"(d.y) : "l"(v));
    return d;
}

__device__ __forceinline__ f32x2 fma2(f32x2 a, f32x2 b, f32x2 c) {
    f32x2 d;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
    return d;
}

__device__ __forceinline__ f32x2 add2(f32x2 a, f32x2 b) {
    f32x2 d;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
    return d;
}

__device__ __forceinline__ f32x2 sub2(f32x2 a, f32x2 b) { return fma2(b, 0xBF800000BF800000ull, a); }  // a - b, rounded once

__device__ __forceinline__ float abs_up(float2 a) { return __fmul_ru(fabsf(a.x), 1.f + 0x1p-22f); }

}  // namespace vbmc
