// ops64.cuh -- FP64 division, square root and the operations on the words of
// a double that the FP64 sweeps use.
//
// The FP64 units take about 80 cycles per warp instruction and scheduler on
// this GPU, so the number of FP64 operations is what bounds the FP64 kernels,
// and integer and FP32 operations are free beside them.  A quotient here
// takes 3 FP64 operations and its reciprocal 2 (shared by all quotients of
// one divisor), a square root 6; a division from the compiler takes about 10
// and a square root about 12.  Both start from a seed of 44 bits formed in
// pairs of floats (a leading part from the special-function unit and its
// residual, by Newton's iteration written out to second order), refined once
// in FP64, and end with the correction step of Markstein (1990), "Computation
// of elementary functions on the IBM RISC System/6000 processor": an exact
// remainder by fused multiply-add, then one fused multiply-add with the
// reciprocal, which rounds correctly.  Operands whose scale could lose bits of
// a remainder (zero, subnormal, huge, not finite) take the compiler's
// operation.
#pragma once
#include "swadj_internal.cuh"

namespace swadj {
namespace d64 {

// ---- the words of a double
__device__ __forceinline__ bool is_zero(double x) {
    return ((__double2hiint(x) << 1) | __double2loint(x)) == 0;
}
__device__ __forceinline__ bool negative(double x) {   // x < 0
    return __double2hiint(x) < 0 && !is_zero(x);
}
__device__ __forceinline__ bool positive(double x) {   // x > 0 (or a positive NaN)
    return __double2hiint(x) >= 0 && !is_zero(x);
}
__device__ __forceinline__ double flip_if(bool neg, double x) {
    return __hiloint2double(__double2hiint(x) ^ (neg ? 0x80000000 : 0), __double2loint(x));
}
__device__ __forceinline__ int exponent(double x) {   // biased, 0 .. 2047
    return (__double2hiint(x) >> 20) & 0x7ff;
}
// x 2^k where neither side leaves the normal numbers
__device__ __forceinline__ double scale(double x, int k) {
    return __hiloint2double(__double2hiint(x) + (k << 20), __double2loint(x));
}
__device__ __forceinline__ double half_of(double x) {
    const int e = exponent(x);
    if (e > 1 && e < 0x7ff) return scale(x, -1);
    return is_zero(x) ? x : 0.5 * x;
}
__device__ __forceinline__ double twice(double x) {
    const int e = exponent(x);
    if (e > 0 && e < 0x7fe) return scale(x, 1);
    return is_zero(x) ? x : 2.0 * x;
}
// smaller and larger of two doubles >= 0
__device__ __forceinline__ double min_pos(double a, double b) {
    return __double_as_longlong(a) < __double_as_longlong(b) ? a : b;
}
__device__ __forceinline__ double max_pos(double a, double b) {
    return __double_as_longlong(a) > __double_as_longlong(b) ? a : b;
}
__device__ __forceinline__ bool is_nan(double x) {
    return (__double_as_longlong(x) & 0x7fffffffffffffffLL) > 0x7ff0000000000000LL;
}

// The mantissa (in [1, 2)) of a normal double as a float of its leading 24
// bits and one of the next 23 (to 2^-47).
__device__ __forceinline__ void split(int hi, int lo, float &h, float &l) {
    h = __uint_as_float(0x3f800000u | ((unsigned)(hi & 0xfffff) << 3) | ((unsigned)lo >> 29));
    const float t = __uint_as_float(0x3f800000u | (((unsigned)lo >> 6) & 0x7fffffu));
    l = (t - 1.f) * 0x1p-23f;
}
// y0 + y1 as a double, y0 in (1/2, 1], |y1| < 2^-20
__device__ __forceinline__ double join(float y0, float y1) {
    const unsigned b = __float_as_uint(y0);
    const long long y =
        ((long long)((b >> 3) + 0x38000000u) << 32) | (long long)((unsigned long long)(b << 29));
    return __longlong_as_double(y + (long long)__float2int_rn(y1 * 0x1p53f));
}

// 1 / b, rounded, for the quotients below; ok = false where b's scale
// is left to the compiler's division.
struct Recip {
    double b, y;
    bool ok;
};
__device__ __forceinline__ Recip recip(double b) {
    Recip r;
    r.b = b;
    const int hi = __double2hiint(b), e = (hi >> 20) & 0x7ff;
    // where 1 / b lies next to a midpoint of two doubles (a mantissa of almost
    // all ones) y may not be its rounding, which the quotients rely on
    r.ok = e > 1023 - 400 && e < 1023 + 400 &&
           !((hi & 0xfffff) == 0xfffff && (unsigned)__double2loint(b) >= 0xfffff000u);
    float h, l;
    split(hi, __double2loint(b), h, l);
    const float y0 = rcp_ftz(h);
    const float q = fmaf(-l, y0, fmaf(-h, y0, 1.f));
    const double m = __hiloint2double((hi & 0xfffff) | 0x3ff00000, __double2loint(b));
    double y = join(y0, y0 * fmaf(q, q, q));
    y = __fma_rn(__fma_rn(-m, y, 1.0), y, y);
    // back to b's scale and sign
    r.y = __hiloint2double((__double2hiint(y) - ((e - 1023) << 20)) ^ (hi & 0x80000000),
                           __double2loint(y));
    return r;
}
// a / b
__device__ __forceinline__ double div(double a, const Recip &r) {
    const int e = exponent(a);
    if (r.ok && e < 1023 + 400 && (e > 1023 - 400 || is_zero(a))) {
        const double q = __dmul_rn(a, r.y);
        return __fma_rn(__fma_rn(-r.b, q, a), r.y, q);
    }
    return a / r.b;
}

__device__ __forceinline__ double root(double a) {
    const int hi = __double2hiint(a), e = hi >> 20;   // negative for a < 0
    if (e > 200 && e < 0x7ff - 200) {
        const int k = (e - 1023) >> 1, odd = (e - 1023) & 1;   // a = m 4^k, m in [1, 4)
        float h, l;
        split(hi, __double2loint(a), h, l);
        if (odd) { h *= 2.f; l *= 2.f; }
        const double m =
            __hiloint2double((hi & 0xfffff) | (0x3ff00000 + (odd << 20)), __double2loint(a));
        const float y0 = rsqrt_ftz(h);
        const float p = y0 * y0, pe = fmaf(y0, y0, -p);
        const float q = fmaf(-l, p, fmaf(-h, pe, fmaf(-h, p, 1.f)));   // 1 - m y0^2
        const double y = join(y0, y0 * fmaf(q * q, 0.375f, 0.5f * q));
        const double z = __fma_rn(__fma_rn(-__dmul_rn(m, y), y, 1.0), scale(y, -1), y);
        const double s = __dmul_rn(m, z);
        return scale(__fma_rn(__fma_rn(-s, s, m), scale(z, -1), s), k);
    }
    return sqrt(a);
}

}  // namespace d64
}  // namespace swadj
