// devmath.cuh -- device helpers shared by the CUDA translation units.
#pragma once
#include <cuda_runtime.h>

namespace ilves {

// float64 -> float32 by truncation, on the integer pipe.  Values below float's normal
// range become signed zero, values above it (never nm-scale coordinates) infinity.
__device__ __forceinline__ float narrow(double v) {
    const unsigned long long b = (unsigned long long)__double_as_longlong(v);
    const unsigned hi = (unsigned)(b >> 32), lo = (unsigned)b;
    const unsigned sign = hi & 0x80000000u;
    const int e = (int)((hi >> 20) & 0x7FFu) - 896;  // rebias 1023 -> 127
    unsigned r = sign | ((unsigned)e << 23) | ((hi & 0xFFFFFu) << 3) | (lo >> 29);
    r = e <= 0 ? sign : r;
    r = e >= 255 ? (sign | 0x7F800000u) : r;
    return __uint_as_float(r);
}

// float32 -> float64, exact, on the integer pipe (subnormal floats flush to zero).
__device__ __forceinline__ double widen(float f) {
    const unsigned b = __float_as_uint(f);
    const unsigned sign = b & 0x80000000u;
    const unsigned e = (b >> 23) & 0xFFu;
    const unsigned mant = b & 0x7FFFFFu;
    unsigned hi = sign | ((e + 896u) << 20) | (mant >> 3);
    unsigned lo = mant << 29;
    hi = e == 0 ? sign : hi;
    lo = e == 0 ? 0u : lo;
    hi = e == 255 ? (sign | 0x7FF00000u | (mant >> 3)) : hi;
    return __hiloint2double((int)hi, (int)lo);
}

// |s| <= t for t >= 0 by comparing bit patterns (NaN compares false)
__device__ __forceinline__ bool abs_le(double s, double t) {
    const long long sb = __double_as_longlong(s) & 0x7FFFFFFFFFFFFFFFll;
    return sb <= __double_as_longlong(t);
}
// |s| <= tol * d2, settled in float32 unless the two are within 2^-20 of each other (or out of
// the middle of float32's range): the float64 product would cost a pipe slot of 66 cycles.
// narrow() truncates, so both float32 values are at most 2^-21 off.
__device__ __forceinline__ bool within(double s, double tol, double d2) {
    const float sf = fabsf(narrow(s)), tf = narrow(tol) * narrow(d2);
    if (tf > 1e-30f && tf < 1e30f) {
        if (sf > tf * (1.0f + 0x1p-20f)) return false;
        if (sf < tf * (1.0f - 0x1p-20f)) return true;
    }
    return abs_le(s, tol * d2);
}
__device__ __forceinline__ bool nonfinite(double s) {
    return (__double_as_longlong(s) & 0x7FF0000000000000ll) == 0x7FF0000000000000ll;
}
__device__ __forceinline__ bool nonfinite(float s) { return (__float_as_uint(s) & 0x7F800000u) == 0x7F800000u; }
__device__ __forceinline__ float lp_abs(float v) { return fabsf(v); }
__device__ __forceinline__ double lp_abs(double v) { return fabs(v); }
// Reciprocal of a pivot.  float32: the hardware approximation and one Newton step by fused
// multiply-adds (Markstein's theorem), the correctly rounded value for every normal a with a
// normal 1 / a (tests/test_gpu_device_math.py compares all 2^32 inputs); about 35 cycles where
// the general routine takes 93.
__device__ __forceinline__ float lp_rcp(float a) {
    const unsigned e = (__float_as_uint(a) >> 23) & 0xFFu;
    if (e - 1u >= 252u) return __frcp_rn(a);  // zero, subnormal, infinite, NaN, or a subnormal result
    float r;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(a));
    return __fmaf_rn(r, __fmaf_rn(-a, r, 1.0f), r);
}
// float64: a float32 seed (relative error below 2^-21) and one step of the third-order iteration
// r (1 + e + e^2), e = 1 - a r (Altman, Pacific J. Math. 10, 1960): three float64 instructions,
// where the division takes about six (a warp's float64 instruction holds its scheduler's pipe for
// 66 cycles on this GPU: 230 against 368 cycles).  The truncated terms are below 2^-63 and the inner
// roundings below 2^-73, so it is at most one ulp from the rounded quotient, and seldom that.
__device__ __forceinline__ double lp_rcp(double a) {
    const int e = (__double2hiint(a) >> 20) & 0x7FF;
    if (e < 1023 - 120 || e > 1023 + 120) return 1.0 / a;
    float s;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(s) : "f"(narrow(a)));
    const double r = widen(s);
    const double d = fma(-a, r, 1.0);
    return fma(r, fma(d, d, d), r);
}
// A pivot s vanished against its assembled entry a: !(|s| > pivot_rel |a|).  float64: settled
// on the exponents alone unless |s| is below about 2^-42 |a|, since a comparison and a product
// in float64 cost two pipe slots of 66 cycles.
template <class Mode>
__device__ __forceinline__ bool pivot_vanished(float s, float a) {
    return !(lp_abs(s) > Mode::pivot_rel * lp_abs(a));
}
template <class Mode>
__device__ __forceinline__ bool pivot_vanished(double s, double a) {
    static_assert(Mode::pivot_rel < 0x1p-43, "the exponent test below");
    const int es = (__double2hiint(s) >> 20) & 0x7FF, ea = (__double2hiint(a) >> 20) & 0x7FF;
    if (es >= ea - 42 && es < 0x7FF && ea < 0x7FF && es > 0) return false;
    return !(lp_abs(s) > Mode::pivot_rel * lp_abs(a));
}

}  // namespace ilves
