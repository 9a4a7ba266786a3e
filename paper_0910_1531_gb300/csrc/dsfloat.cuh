// Double-single arithmetic: a value as the unevaluated sum hi + lo of two floats, |lo| <= ulp(hi) / 2
// (about 48 significant bits), by Knuth's TwoSum and the FMA product error (Dekker 1971; Knuth, The
// Art of Computer Programming 4.2.2).  The grand-potential sums of FP32 plans use it: their terms are
// functions of FP32 fields, and the FP64 pipe of the GPU has 1/64 of the FP32 rate.
//
// Every operation uses the _rn intrinsics, which the compiler does not contract.
#pragma once

#include <cuda_runtime.h>

namespace dftk {

struct ds {
    float hi, lo;
};

__device__ __forceinline__ ds ds_sum2(float a, float b) {      // a + b exactly
    const float s = __fadd_rn(a, b), bb = __fsub_rn(s, a);
    return {s, __fadd_rn(__fsub_rn(a, __fsub_rn(s, bb)), __fsub_rn(b, bb))};
}
__device__ __forceinline__ ds ds_norm(float a, float b) {      // the same where |a| >= |b|
    const float s = __fadd_rn(a, b);
    return {s, __fsub_rn(b, __fsub_rn(s, a))};
}
__device__ __forceinline__ ds ds_prod2(float a, float b) {     // a b exactly
    const float p = __fmul_rn(a, b);
    return {p, __fmaf_rn(a, b, -p)};
}
__device__ __forceinline__ ds operator+(ds a, ds b) {
    const ds s = ds_sum2(a.hi, b.hi);
    return ds_norm(s.hi, __fadd_rn(s.lo, __fadd_rn(a.lo, b.lo)));
}
__device__ __forceinline__ ds operator-(ds a) { return {-a.hi, -a.lo}; }
__device__ __forceinline__ ds operator-(ds a, ds b) { return a + (-b); }
__device__ __forceinline__ ds operator*(ds a, ds b) {
    const ds p = ds_prod2(a.hi, b.hi);
    return ds_norm(p.hi, __fmaf_rn(a.hi, b.lo, __fmaf_rn(a.lo, b.hi, p.lo)));
}
__device__ __forceinline__ ds operator*(ds a, float b) {
    const ds p = ds_prod2(a.hi, b);
    return ds_norm(p.hi, __fmaf_rn(a.lo, b, p.lo));
}
__device__ __forceinline__ ds ds_recip(ds a) {                 // one Newton step from the float reciprocal
    const float r = __frcp_rn(a.hi);
    const float e = __fmaf_rn(-a.lo, r, __fmaf_rn(-a.hi, r, 1.0f));
    const float c = __fmul_rn(r, e);
    return ds_norm(r, __fmaf_rn(c, e, c));
}
// a constant rounded to a pair
__host__ __device__ constexpr ds ds_const(double v) { return {float(v), float(v - double(float(v)))}; }

// ln(a) for 1e-30 < a.hi < 1e30: a.hi = 2^k m with m in [sqrt(1/2), sqrt(2)), and with
// s = (m - 1) / (m + 1), ln m = 2 s (1 + s^2 / 3 + s^4 / 5 + ...) (the series of the inverse
// hyperbolic tangent), its first terms in pairs and the rest, below 2.6e-5 of the sum, in float;
// a.lo adds ln(1 + a.lo / a.hi) to second order.  Error below 1e-12 max(1, |ln a|) (6e-13 over 3e6
// arguments against FP64), where a logarithm of FP32 fields enters sums of FP32 accuracy.
__device__ __forceinline__ ds ds_log(ds a) {
    const int bits = __float_as_int(a.hi);
    int k = (bits - 0x3f3504f3) >> 23;
    const float m = __int_as_float(bits - (k << 23));
    const ds s = ds_norm(__fsub_rn(m, 1.0f), 0.0f) * ds_recip(ds_sum2(m, 1.0f));
    const ds z = s * s;
    const float zf = z.hi;
    float q = 1.0f / 21;
    q = __fmaf_rn(q, zf, 1.0f / 19);
    q = __fmaf_rn(q, zf, 1.0f / 17);
    q = __fmaf_rn(q, zf, 1.0f / 15);
    q = __fmaf_rn(q, zf, 1.0f / 13);
    q = __fmaf_rn(q, zf, 1.0f / 11);
    q = __fmaf_rn(q, zf, 1.0f / 9);
    ds t = z * q + ds_const(1.0 / 7);
    t = z * t + ds_const(1.0 / 5);
    t = z * t + ds_const(1.0 / 3);
    ds r = s + s * (z * t);
    r = {2.0f * r.hi, 2.0f * r.lo};
    r = r + ds_const(0.69314718055994530942) * float(k);
    const float l = __fdiv_rn(a.lo, a.hi);
    return r + ds{__fmaf_rn(-0.5f * l, l, l), 0.0f};
}

}  // namespace dftk
