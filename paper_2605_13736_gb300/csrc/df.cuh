// Double-float arithmetic on the FP32 pipes: a value is s + c, c of the order
// of 2^-24 s (gemv_df.cu explains the products and their accuracy).
#pragma once

namespace mdsip {

// (s, c) += a x in double-float, a = (ah, al), x = (xh, xl)
__device__ __forceinline__ void df_acc(float ah, float al, float xh, float xl, float &s, float &c) {
    const float p = ah * xh;
    const float pe = fmaf(ah, xh, -p);                 // exact error of the product
    const float sm = fmaf(ah, xl, fmaf(al, xh, pe));   // the small terms (al xl dropped: 2^-48)
    const float t = s + p;                             // two-sum (Knuth): s + p = t + e exactly
    const float bb = t - s;
    const float e = (s - (t - bb)) + (p - bb);
    s = t;
    c += e + sm;
}

__device__ __forceinline__ void df_add(float &s, float &c, float s2, float c2) {
    const float t = s + s2, bb = t - s;
    const float e = (s - (t - bb)) + (s2 - bb);
    s = t;
    c = c + c2 + e;
}

// df_acc on two lanes at once with the packed FP32 instructions (each lane
// rounded exactly as the scalar form; a - b as fma(b, -1, a))
__device__ __forceinline__ void df_acc2(float2 ah, float2 al, float2 xh, float2 xl, float2 &s, float2 &c) {
    const float2 m1 = make_float2(-1.0f, -1.0f);
    const float2 p = __fmul2_rn(ah, xh);
    const float2 pe = __ffma2_rn(ah, xh, __fmul2_rn(p, m1));           // exact error of the product
    const float2 sm = __ffma2_rn(ah, xl, __ffma2_rn(al, xh, pe));       // the small terms
    const float2 t = __fadd2_rn(s, p);                                  // two-sum: s + p = t + e
    const float2 bb = __ffma2_rn(s, m1, t);
    const float2 e = __fadd2_rn(__ffma2_rn(__ffma2_rn(bb, m1, t), m1, s), __ffma2_rn(bb, m1, p));
    s = t;
    c = __fadd2_rn(c, __fadd2_rn(e, sm));
}

}  // namespace mdsip
