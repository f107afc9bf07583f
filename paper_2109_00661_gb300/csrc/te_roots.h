// Vertical wavenumbers and interface coefficients of the FP32 TE recursion, two
// abscissae at a time (forward.cu, adjoint.cu; the form and its accuracy are
// described in forward.cu).
#pragma once

#include "f32x2.h"

namespace aem {
namespace f32x2 {

struct Root {  // w of one layer for both abscissae, and m = |w|^2 / 2
    u64 re, im, m;
};

// rec = ((Re s, Re s), (Im s, Im s)).
__device__ __forceinline__ Root root2(u64 lam2, ulonglong2 rec) {
    const u64 x = add2(lam2, rec.x);
    const u64 v = fma2(x, x, mul2(rec.y, rec.y));
    float v0, v1, x0, x1;
    up2(v, v0, v1);
    up2(x, x0, x1);
    const float m0 = sqrt_approx(v0), m1 = sqrt_approx(v1);
    const float t0 = m0 + fabsf(x0), t1 = m1 + fabsf(x1);
    const u64 rr = pk2(rsqrt_approx(t0), rsqrt_approx(t1));
    const u64 p = mul2(pk2(t0, t1), rr), o = mul2(rec.y, rr);
    Root w;
    w.m = pk2(m0, m1);
    float p0, p1, o0, o1;
    up2(p, p0, p1);
    up2(o, o0, o1);
    w.re = pk2(x0 >= 0.f ? p0 : o0, x1 >= 0.f ? p1 : o1);
    w.im = pk2(x0 >= 0.f ? o0 : p0, x1 >= 0.f ? o1 : p1);
    return w;
}

// 1 / d for both abscissae from one reciprocal: three multiplications in place
// of the second special-function operation (the layer-step's busiest unit;
// marginal layer 98.8 -> 96.7 SM-sub-partition cycles per 32 items).
__device__ __forceinline__ u64 rcp2(u64 d) {
    float d0, d1;
    up2(d, d0, d1);
    const float i = rcp_approx(d0 * d1);
    return pk2(i * d1, i * d0);
}

// The interface coefficient between a (above) and b.
__device__ __forceinline__ C2x2 rcoef2(const Root &a, const Root &b) {
    const u64 den = fma2(a.im, b.im, fma2(a.re, b.re, add2(a.m, b.m)));
    const u64 ir = rcp2(den);
    C2x2 r;
    r.re = mul2(sub2(a.m, b.m), ir);
    r.im = mul2(sub2(mul2(a.im, b.re), mul2(a.re, b.im)), ir);
    return r;
}

}  // namespace f32x2
}  // namespace aem
