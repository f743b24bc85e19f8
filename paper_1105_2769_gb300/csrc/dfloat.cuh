// Numbers carried as an unevaluated sum of two FP32 values (about 2^-46 relative),
// from exact sums and FMA products: pair terms that FP64, at 1/64 of the FP32
// rate, would make the longest part of a pass.
#pragma once

#include <cuda_runtime.h>

struct df {
    float h, l;
};
__device__ __forceinline__ df df_fast(float a, float b) {  // |a| >= |b|
    const float s = __fadd_rn(a, b);
    return {s, __fsub_rn(b, __fsub_rn(s, a))};
}
__device__ __forceinline__ df df_mul(df a, df b) {
    const float p = __fmul_rn(a.h, b.h);
    float e = __fmaf_rn(a.h, b.h, -p);
    e = __fmaf_rn(a.h, b.l, e);
    e = __fmaf_rn(a.l, b.h, e);
    return df_fast(p, e);
}
__device__ __forceinline__ df df_add(df a, df b) {
    const float s = __fadd_rn(a.h, b.h);
    const float t = __fsub_rn(s, a.h);
    float e = __fadd_rn(__fsub_rn(a.h, __fsub_rn(s, t)), __fsub_rn(b.h, t));
    e = __fadd_rn(e, __fadd_rn(a.l, b.l));
    return df_fast(s, e);
}
__device__ __forceinline__ df df_diff(float qh, float ql, float ph, float pl) {
    const float s = __fsub_rn(qh, ph);
    const float t = __fsub_rn(s, qh);
    const float e = __fsub_rn(__fsub_rn(qh, __fsub_rn(s, t)), __fadd_rn(ph, t));
    return df_fast(s, __fadd_rn(e, __fsub_rn(ql, pl)));
}

// a . b of two 3-vectors.
__device__ __forceinline__ df df_dot(const df (&a)[3], const df (&b)[3]) {
    float s = __fmul_rn(a[0].h, b[0].h);
    float e = __fmaf_rn(a[0].h, b[0].h, -s);
    e = __fmaf_rn(a[0].h, b[0].l, e);
    e = __fmaf_rn(a[0].l, b[0].h, e);
#pragma unroll
    for (int d = 1; d < 3; ++d) {
        const float p = __fmul_rn(a[d].h, b[d].h);
        float pe = __fmaf_rn(a[d].h, b[d].h, -p);
        pe = __fmaf_rn(a[d].h, b[d].l, pe);
        pe = __fmaf_rn(a[d].l, b[d].h, pe);
        const float t = __fadd_rn(s, p), u = __fsub_rn(t, s);
        e = __fadd_rn(e, __fadd_rn(pe, __fadd_rn(__fsub_rn(s, __fsub_rn(t, u)), __fsub_rn(p, u))));
        s = t;
    }
    return df_fast(s, e);
}

// 1/sqrt(s): hardware estimate and one Newton step kept as a two-term number.
__device__ __forceinline__ df df_rsqrt(df s) {
    const float y0 = rsqrtf(s.h);
    const float p = __fmul_rn(y0, y0), pe = __fmaf_rn(y0, y0, -p);
    const float q = __fmul_rn(s.h, p), qe = __fmaf_rn(s.h, p, -q);
    const float res =
        __fsub_rn(__fsub_rn(1.0f, q), __fmaf_rn(s.l, p, __fmaf_rn(s.h, pe, qe)));
    return df_fast(y0, __fmul_rn(__fmul_rn(0.5f, y0), res));
}
