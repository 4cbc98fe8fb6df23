// bq_pairs.cuh -- double-float sums of products on pairs of values (the packed FP32
// instructions of the sm_100 family), shared by the hopping kernels and the gauge-side ones.
#pragma once

#include "bq_device.cuh"

// Lazy double-float sums of products on (real, imaginary) pairs with the packed
// FP32 instructions of the sm_100 family (one instruction for both lanes): lane x
// and lane y take exactly the operations of two scalar dfsum chains.
struct dfsum2 {
    float2 s, c;
};
__device__ __forceinline__ float2 f2neg(float2 a) { return make_float2(-a.x, -a.y); }
__device__ __forceinline__ dfsum2 dfs2_prod(float2 ah, float2 al, float2 bh, float2 bl) {
    const float2 p = __fmul2_rn(ah, bh);
    float2 e = __ffma2_rn(ah, bh, f2neg(p));
    e = __ffma2_rn(ah, bl, e);
    e = __ffma2_rn(al, bh, e);
    return {p, e};
}
__device__ __forceinline__ void dfs2_add_prod(dfsum2 &z, float2 ah, float2 al, float2 bh, float2 bl) {
    const float2 p = __fmul2_rn(ah, bh);
    float2 e = __ffma2_rn(ah, bh, f2neg(p));
    e = __ffma2_rn(ah, bl, e);
    e = __ffma2_rn(al, bh, e);
    // two-sum of z.s and p
    const float2 t = __fadd2_rn(z.s, p);
    const float2 bb = __fadd2_rn(t, f2neg(z.s));
    const float2 te = __fadd2_rn(__fadd2_rn(z.s, f2neg(__fadd2_rn(t, f2neg(bb)))), __fadd2_rn(p, f2neg(bb)));
    z.s = t;
    z.c = __fadd2_rn(z.c, __fadd2_rn(e, te));
}

// a + b = s + c, error-free
__device__ __forceinline__ dfsum2 two_sum2(float2 a, float2 b) {
    const float2 t = __fadd2_rn(a, b);
    const float2 bb = __fadd2_rn(t, f2neg(a));
    return {t, __fadd2_rn(__fadd2_rn(a, f2neg(__fadd2_rn(t, f2neg(bb)))), __fadd2_rn(b, f2neg(bb)))};
}
// the normalised value of a sum (dfs_done of both)
__device__ __forceinline__ void dfs2_done(dfsum2 z, float2 &hi, float2 &lo) {
    const dfsum2 t = two_sum2(z.s, z.c);
    hi = __fadd2_rn(t.s, t.c);
    lo = __fadd2_rn(t.c, f2neg(__fadd2_rn(hi, f2neg(t.s))));
}
