// Scalar helpers with few FP64 operations: a warp's FP64 instruction takes 64
// clocks of its scheduler on this GPU however few lanes are active, so scalings by
// powers of two are exponent arithmetic, and roots and reciprocals are one step of
// Householder's third-order iteration (A. S. Householder, The Numerical Treatment of
// a Single Nonlinear Equation, 1970) from an FP32 seed: with the seed's residual t,
// the series of (1 - t)^(-1/2) or (1 - t)^(-1) through t^2.
#pragma once

#include "common.cuh"

namespace sim {

// 1 / sqrt(d) for a d well inside the range of normal numbers: an FP32 seed y0 of
// d scaled by an even power of two, then y0 + y0 t (1/2 + 3/8 t) with t = 1 - d y0^2
// (five FP64 operations; the seed's 2^-22 leaves less than 2^-60).
__device__ __forceinline__ double rsqrt_nr(double d) {
    const uint32_t hd = (uint32_t)__double2hiint(d), ld = (uint32_t)__double2loint(d);
    const int e = ((int)(hd >> 20) - 1023) & ~1;  // even; d 2^-e in [1, 4)
    const float f = __uint_as_float((((hd >> 20) - 1023u - (uint32_t)e + 127u) << 23) | ((hd & 0xFFFFFu) << 3) | (ld >> 29));
    const uint32_t g = __float_as_uint(rsqrtf(f));  // (0.5, 1]
    const double y0 = __hiloint2double((int)((((g >> 23) - 127u + 1023u - (uint32_t)(e / 2)) << 20) | ((g & 0x7FFFFFu) >> 3)),
                                       (int)(g << 29));
    const double t = fma(-(d * y0), y0, 1.0);
    return fma(y0 * t, fma(0.375, t, 0.5), y0);
}

// float <-> double by integer arithmetic: the conversion instructions go through
// the FP64 pipe.  Same values, rounded to nearest even; what is not a normal number
// on both sides (zero apart) takes the instruction.
__device__ __forceinline__ double widen(float f) {
    const uint32_t b = __float_as_uint(f), e = (b >> 23) & 255u;
    if ((b << 1) == 0u) return __hiloint2double((int)b, 0);
    if (e == 0u || e == 255u) return (double)f;
    return __hiloint2double((int)((b & 0x80000000u) | (((b & 0x7FFFFFFFu) >> 3) + (896u << 20))), (int)(b << 29));
}
__device__ __forceinline__ float narrow(double d) {
    const uint32_t h = (uint32_t)__double2hiint(d), l = (uint32_t)__double2loint(d);
    const uint32_t e = (h >> 20) & 2047u;
    if (((h << 1) | l) == 0u) return __uint_as_float(h);
    if (e < 898u || e > 1149u) return (float)d;
    uint32_t m = (((h & 0x7FFFFFFFu) - (896u << 20)) << 3) | (l >> 29);
    const uint32_t rest = l & 0x1FFFFFFFu;
    m += (rest > 0x10000000u || (rest == 0x10000000u && (m & 1u))) ? 1u : 0u;
    return __uint_as_float((h & 0x80000000u) | m);
}
__device__ __forceinline__ float2 narrow(double2 v) { return make_float2(narrow(v.x), narrow(v.y)); }
__device__ __forceinline__ double2 widen(float2 v) { return make_double2(widen(v.x), widen(v.y)); }

// v 2^k, zero where v or the result is zero or subnormal
__device__ __forceinline__ double scale2(double v, int k) {
    const uint32_t h = (uint32_t)__double2hiint(v);
    const int e = (int)((h >> 20) & 2047u);
    return e > 0 && e + k > 0 ? __hiloint2double((int)(h + ((uint32_t)k << 20)), __double2loint(v)) : 0.0;
}

// 1 / a far out of the middle of the range, e its exponent: by division.  A function of
// its own, so that its rare code does not lie in the pivot chains' loops.
static __device__ __noinline__ double2 crecip_far(double2 a, int e) {
    if (isinf(a.x) || isinf(a.y)) return make_double2(0.0, 0.0);
    const double s = e < 64 ? 0x1p+960 : 0x1p-960;
    const double x = a.x * s, y = a.y * s, d = x * x + y * y;
    return make_double2(x / d * s, -(y / d) * s);
}

// 1 / a (seven FP64 operations): 1/d, d = |a 2^k|^2 in [1, 8), is r + r (e + e^2) with
// e = 1 - d r from an FP32 reciprocal r (2 ulp: e^3 < 2^-60).
__device__ __forceinline__ double2 crecip(double2 a) {
    const int e = max((__double2hiint(a.x) >> 20) & 2047, (__double2hiint(a.y) >> 20) & 2047);
    if (e < 64 || e > 1983) return crecip_far(a, e);
    const int k = 1023 - e;  // a 2^k has its larger part in [1, 2)
    const double x = scale2(a.x, k), y = scale2(a.y, k);
    const double d = fma(x, x, y * y);  // [1, 8)
    const uint32_t hd = (uint32_t)__double2hiint(d), ld = (uint32_t)__double2loint(d);
    const float f = __uint_as_float(((((hd >> 20) & 2047u) - 1023u + 127u) << 23) | ((hd & 0xFFFFFu) << 3) | (ld >> 29));
    const uint32_t g = __float_as_uint(__fdividef(1.0f, f));
    const double r0 = __hiloint2double((int)((((g >> 23) - 127u + 1023u) << 20) | ((g & 0x7FFFFFu) >> 3)), (int)(g << 29));
    const double t = fma(-d, r0, 1.0);
    const double r = fma(r0, fma(t, t, t), r0);
    return make_double2(scale2(x * r, k), scale2(-(y * r), k));
}

// The same in FP32: a division's seed and one Newton step.  The power of two goes
// onto the components, not onto the real reciprocal, which it could overflow.
__device__ __forceinline__ float2 crecip(float2 a) {
    const float m = fmaxf(fabsf(a.x), fabsf(a.y));
    const int e = (int)((__float_as_uint(m) >> 23) & 255u);
    const float s = __uint_as_float((uint32_t)min(max(254 - e, 1), 253) << 23);  // about 1/m
    const float x = a.x * s, y = a.y * s;  // the larger in [1, 2) but for the ends of the range
    const float d = fmaf(x, x, y * y);
    float r = __fdividef(1.0f, d);
    r = fmaf(r, fmaf(-d, r, 1.0f), r);  // one Newton step
    return make_float2((x * s) * r, -((y * s) * r));
}

}  // namespace sim
