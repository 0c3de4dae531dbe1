// FP32 evaluation of the exponential-of-semicircle spreading function by the hardware
// approximations (the ring kernels' kernel values).
#pragma once
#include "common.cuh"

namespace nlp {

// exp(beta (sqrt(1 - x^2) - 1)) for x = (i - d) 2/w with the exponent written as
// -beta x^2 / (1 + sqrt(1 - x^2)) (no cancellation near x = 0); 0 outside |x| < 1.
// nbl2 = -beta log2(e).  rsqrt / rcp / ex2 are the hardware approximations.
__device__ __forceinline__ float es_fast(float i_f, float d, float c2w, float nbl2) {
    const float x = (i_f - d) * c2w;
    const float s = fmaf(-x, x, 1.0f);
    float rs, rd, e;
    asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(rs) : "f"(s));
    const float den = fmaf(s, rs, 1.0f);
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(rd) : "f"(den));
    const float arg = (x * (x * nbl2)) * rd;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(e) : "f"(arg));
    return s > 0.0f ? e : 0.0f;
}

__device__ __forceinline__ float2 f2(float a, float b) { return make_float2(a, b); }

// es_fast for two values at once: the same operations, the FP32 ones as packed FP32x2 (each
// lane of a packed operation rounds as the scalar one), the approximations per value.
__device__ __forceinline__ float2 es_fast2(float2 i_f, float2 d, float c2w, float nbl2) {
    const float2 x = __fmul2_rn(__fadd2_rn(i_f, f2(-d.x, -d.y)), f2(c2w, c2w));
    const float2 s = __ffma2_rn(f2(-x.x, -x.y), x, f2(1.0f, 1.0f));
    float2 rs, rd, e;
    asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(rs.x) : "f"(s.x));
    asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(rs.y) : "f"(s.y));
    const float2 den = __ffma2_rn(s, rs, f2(1.0f, 1.0f));
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(rd.x) : "f"(den.x));
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(rd.y) : "f"(den.y));
    const float2 arg = __fmul2_rn(__fmul2_rn(x, __fmul2_rn(x, f2(nbl2, nbl2))), rd);
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(e.x) : "f"(arg.x));
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(e.y) : "f"(arg.y));
    return f2(s.x > 0.0f ? e.x : 0.0f, s.y > 0.0f ? e.y : 0.0f);
}

}  // namespace nlp
