// The projection's reciprocal norm of the unrolled solver, on packed FP32 pairs.
#pragma once

#include "tv_body.cuh"

namespace cslsm {

__device__ __forceinline__ float2 splat(float v) { return make_float2(v, v); }

// 1 / max(1, sqrt(s)) of a pair.  Square root and reciprocal by Markstein's FMA residual
// corrections (P. Markstein, "IA-64 and Elementary Functions", 2000) of the approximate
// reciprocal root, packed and free of branches: sqrtf and the division take a slow-path
// branch each, which keeps a warp's rows from overlapping (unrolled forward of 8 x 16 x
// 512 x 512, 5 iterations: 15.6 against 11.3 ms).  The reciprocal starts one ulp high,
// which settles the roots with an all-ones mantissa.  For every finite s >= 1 the result
// equals 1.f / sqrtf(s) (all 2^30 of them compared on this GPU; a test compares every
// mantissa of two exponents and a sample of the others): the iterates of the unrolled
// solver stand on the kink of the projection, where one ulp can flip a gradient's
// branch.  Infinity gives 0 and NaN gives 1, as 1.f / fmaxf(1.f, sqrtf(s)) does.
__device__ __forceinline__ float2 inv_norm2(float2 s)
{
    const float2 m = make_float2(fmaxf(s.x, 1.f), fmaxf(s.y, 1.f));
    float2 y;
    asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(y.x) : "f"(m.x));
    asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(y.y) : "f"(m.y));
    const float2 g = mul2(m, y), ng = mul2(m, mul2(y, splat(-1.f)));
    const float2 r = fma2(ng, g, m);                           // m - g^2, exact
    const float2 nroot = fma2(r, mul2(y, splat(-0.5f)), ng);   // -sqrt(m)
    const float2 yb = fma2(y, splat(1.1920929e-7f), y);
    const float2 e = fma2(nroot, yb, splat(1.f));
    const float2 x = fma2(e, fma2(e, yb, yb), yb);
    return make_float2(fmaxf(x.x, 0.f), fmaxf(x.y, 0.f));  // NaN (overflow) to 0
}

}  // namespace cslsm
