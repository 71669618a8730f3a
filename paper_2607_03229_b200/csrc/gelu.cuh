// GELU (u Phi(u), erf form) and its derivative as the projection epilogues evaluate them, two values at a time in packed fp32.
#pragma once
#include "sm100_ptx.cuh"

namespace mpipe {

// What both need of u: e = exp(-u^2 / 2) and s = erf(u / sqrt 2), by the rational-times-Gaussian form of Abramowitz & Stegun
// 7.1.26 (|error| <= 1.5e-7, far below the bf16 rounding of the result): erf(x) = 1 - (a1 t + ... + a5 t^5) exp(-x^2) with
// t = 1 / (1 + 0.3275911 x), x >= 0.  The Gaussian is the density the derivative needs as well: one exponential and one
// reciprocal per value in either function.
__device__ __forceinline__ float2 splat2(float a) { return make_float2(a, a); }
__device__ __forceinline__ void erf_gauss2(float2 u, float2& erf, float2& gauss) {
    const float2 au = make_float2(fabsf(u.x), fabsf(u.y));
    const float2 d = fma2(au, splat2(0.3275911f * 0.7071067811865476f), splat2(1.0f));
    float2 t;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(t.x) : "f"(d.x));
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(t.y) : "f"(d.y));
    const float2 x = mul2(mul2(u, splat2(-0.5f * 1.4426950408889634f)), u);
    gauss = make_float2(ex2_approx(x.x), ex2_approx(x.y));
    float2 p = fma2(splat2(-1.061405429f), t, splat2(1.453152027f));   // the negated polynomial
    p = fma2(p, t, splat2(-1.421413741f));
    p = fma2(p, t, splat2(0.284496736f));
    p = fma2(p, t, splat2(-0.254829592f));
    const float2 r = fma2(mul2(p, t), gauss, splat2(1.0f));
    erf = make_float2(copysignf(r.x, u.x), copysignf(r.y, u.y));
}
__device__ __forceinline__ float2 gelu_erf2(float2 u) {
    float2 s, e;
    erf_gauss2(u, s, e);
    const float2 h = mul2(u, splat2(0.5f));
    return fma2(h, s, h);
}
// d/du [u Phi(u)] = Phi(u) + u phi(u), phi the standard normal density
__device__ __forceinline__ float2 gelu_erf_grad2(float2 u) {
    float2 s, e;
    erf_gauss2(u, s, e);
    const float2 cdf = fma2(s, splat2(0.5f), splat2(0.5f));
    return fma2(mul2(u, splat2(0.3989422804014327f)), e, cdf);
}

}  // namespace mpipe
