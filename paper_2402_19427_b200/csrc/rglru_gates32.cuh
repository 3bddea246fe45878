// Gate and decay arithmetic of Eq. 1-4 at fp32 accuracy (1-2 units in the last place) on packed pairs: what the kernels use whose
// callers are promised fp32 throughout.  Device code only.
// With the library's expf, expm1f, sqrtf and a divide these are about ninety instructions per element, which alone took 20 us on
// B5 T1021 D1536; here they are about twenty-five, most of them on two elements at once.
#pragma once

#include "rglru_internal.h"
#include "sm100_gates.cuh"

namespace rglru {

__device__ __forceinline__ float rsqrt_approx(float x) { float y; asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x)); return y; }
__device__ __forceinline__ float clamp_nan(float z, float lim) {   // to [-lim, lim]; a NaN stays one
    float y;
    asm("{\n.reg .f32 t;\nmin.NaN.f32 t, %1, %2;\nmax.NaN.f32 %0, t, %3;\n}" : "=f"(y) : "f"(z), "f"(lim), "f"(-lim));
    return y;
}
// 1 / (1 + exp(-z)).  The exponent -z log2(e) is carried with its rounding error, the reciprocal gets one Newton step; beyond +-87 the
// result is 0 or 1 to fp32 anyway, and exp(87) is still finite.
__device__ __forceinline__ f32x2 sigmoid2_acc(f32x2 z) {
    const f32x2 n = pack2(clamp_nan(-z.x, 87.0f), clamp_nan(-z.y, 87.0f)), ONE = pack2(1.0f, 1.0f);
    const f32x2 hi = pack2(1.44269502f, 1.44269502f), lo = pack2(1.92596303e-8f, 1.92596303e-8f), ln2 = pack2(0.693147181f, 0.693147181f);
    const f32x2 t = mul2(n, hi);
    const f32x2 rest = fma2(n, lo, fma2(n, hi, mul2(t, pack2(-1.0f, -1.0f))));
    const f32x2 e0 = pack2(ex2_approx(t.x), ex2_approx(t.y));
    const f32x2 q = __fadd2_rn(fma2(mul2(e0, ln2), rest, e0), ONE);
    const f32x2 r0 = pack2(rcp_approx(q.x), rcp_approx(q.y));
    return fma2(r0, fma2(mul2(q, pack2(-1.0f, -1.0f)), r0, ONE), r0);
}
// f = 1 - a_t = 1 - exp(-s r) of Eq. 3 without cancellation.  POLY: s <= S_POLY for both (and r <= 1)
template <bool POLY> __device__ __forceinline__ f32x2 one_minus_decay2(f32x2 r, f32x2 s) {
    const f32x2 x = mul2(r, s);
    if (POLY) {   // x - x^2/2 + x^3/6 - ... - x^6/720: relative truncation error below 5e-8
        f32x2 p = fma2(x, pack2(-1.0f / 720.0f, -1.0f / 720.0f), pack2(1.0f / 120.0f, 1.0f / 120.0f));
        p = fma2(p, x, pack2(-1.0f / 24.0f, -1.0f / 24.0f));
        p = fma2(p, x, pack2(1.0f / 6.0f, 1.0f / 6.0f));
        p = fma2(p, x, pack2(-0.5f, -0.5f));
        return fma2(mul2(p, x), x, x);
    }
    return pack2(-expm1f(-x.x), -expm1f(-x.y));
}
// m = sqrt(1 - a_t^2) = sqrt(f (2 - f)) and, on the way, 1 / m.  Below m = 1e-15 (where r is below 1e-29) both are only bounded: m by
// 1e-15, 1 / m by 1e15
__device__ __forceinline__ f32x2 input_scale2(f32x2 f, f32x2 &rm) {
    const f32x2 q = mul2(f, fma2(f, pack2(-1.0f, -1.0f), pack2(2.0f, 2.0f)));
    const f32x2 y = pack2(rsqrt_approx(fmaxf(q.x, 1e-30f)), rsqrt_approx(fmaxf(q.y, 1e-30f)));
    const f32x2 m0 = mul2(q, y), hy = mul2(y, pack2(0.5f, 0.5f));
    rm = fma2(hy, fma2(mul2(m0, pack2(-1.0f, -1.0f)), y, pack2(1.0f, 1.0f)), y);           // y (3 - q y^2) / 2
    return fma2(fma2(mul2(m0, pack2(-1.0f, -1.0f)), m0, q), hy, m0);
}

// s = c softplus(-Lambda)   (Appendix A, with a = sigmoid(Lambda))
__device__ __forceinline__ float decay_rate_acc(float lambda, float c) {
    const float z = -lambda;
    return c * (z > 0.0f ? z + log1pf(expf(-z)) : log1pf(expf(z)));
}

// GeLU(v) = v Phi(v), the non-linearity on the second branch of the recurrent block (Section 2.3).  Below -64 Phi(v) is 0 in fp32, and
// -64 stands in for v: -infinity times that 0 would be NaN
__device__ __forceinline__ float gelu_acc(float v) {
    v = v < -64.0f ? -64.0f : v;
    return 0.5f * v * (1.0f + erff(v * 0.70710678f));
}

}  // namespace rglru
