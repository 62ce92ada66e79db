// ops64.cuh -- FP64 division, square root and the operations on the words of
// a double that the FP64 sweeps use.
//
// The FP64 units take about 80 cycles per warp instruction and scheduler on
// this GPU, so the number of FP64 operations is what bounds the FP64 kernels,
// and integer and FP32 operations run beside them.  Quotients and square
// roots take no FP64 operation here (a division from the compiler about 10, a
// square root about 12): a seed of 44 bits formed in pairs of floats (a
// leading part from the special-function unit and its residual, by Newton's
// iteration written out to second order) is refined once as a 64-bit fixed
// point number, and gives a quotient (root) that is the integer below the
// exact one or the next below that.  The exact remainder, an integer of less
// than 57 bits, decides the rounding: no quotient of two 53-bit numbers and
// no square root of one lies half way between two 53-bit numbers.  Operands
// that are subnormal or not finite, and quotients outside the normal numbers or
// beside their ends, take the compiler's operation.  Every other scale counts:
// the front of a wave that spreads into the ocean at rest falls off by orders
// of magnitude a cell, and the limiter divides products of two such values.
// With operands within 2^-400 to 2^400 only, the warps there ran the compiler's
// division beside this one.
// Measured, us per step from a source at rest, so / now: forward 128^2 100 / 83
// (the tiled kernel 83), 512^2 183 / 138, 1024^2 332 / 256, with waves everywhere
// 272 / 270 at 512^2; adjoint 512^2 109 / 98.  A zero dividend is left to the end,
// out of every other quotient's way (wet/dry 511 x 350 254 / 251).
// A quotient takes about 40 integer instructions, the reciprocal that all
// quotients of one divisor share 30, a root 55.
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

// (float)x, to nearest even.  The hardware's conversion goes through the FP64
// units, which bound the kernel that sets an FP32 state from FP64 arrays.
__device__ __forceinline__ float to_float(double x) {
    const int hi = __double2hiint(x), e = (hi >> 20) & 0x7ff;
    const unsigned lo = (unsigned)__double2loint(x), sign = (unsigned)hi & 0x80000000u;
    if (e >= 897 && e <= 1150) {   // from the smallest normal float; may round to infinity
        unsigned b = (((unsigned)hi & 0x7fffffffu) - (896u << 20)) << 3 | lo >> 29;
        const unsigned rest = lo << 3;   // the bits below, 2^31 one half
        b += rest > 0x80000000u || (rest == 0x80000000u && (b & 1));
        return __uint_as_float(b | sign);
    }
    if (is_zero(x)) return __uint_as_float(sign);
    return (float)x;
}

// The mantissa (in [1, 2)) of a normal double as a float of its leading 24
// bits and one of the next 23 (to 2^-47).
__device__ __forceinline__ void split(int hi, int lo, float &h, float &l) {
    h = __uint_as_float(0x3f800000u | ((unsigned)(hi & 0xfffff) << 3) | ((unsigned)lo >> 29));
    const float t = __uint_as_float(0x3f800000u | (((unsigned)lo >> 6) & 0x7fffffu));
    l = (t - 1.f) * 0x1p-23f;
}
// (y0 + y1) 2^63, y0 in [1/2, 1], |y1| < 2^-20, to 2^13
__device__ __forceinline__ unsigned long long join(float y0, float y1) {
    return ((unsigned long long)(__float_as_uint(y0) - 0x3e800000u) << 39) +
           (unsigned long long)((long long)__float2int_rn(y1 * 0x1p50f) << 13);
}
// y + y d 2^-(32 + k), d a correction of few bits
__device__ __forceinline__ unsigned long long refine(unsigned long long y, int d, int k) {
    return y + (unsigned long long)(((long long)(unsigned)(y >> 32) * (long long)d) >> k);
}
// The mantissa of a normal double as an integer in [2^52, 2^53).
__device__ __forceinline__ unsigned long long mantissa(double x) {
    return ((unsigned long long)(((unsigned)__double2hiint(x) & 0xfffffu) | 0x100000u) << 32) |
           (unsigned)__double2loint(x);
}

// A divisor b: y, 1 to 6 units below 2^63 2^52 / mantissa (2^52 / mantissa is in
// (1/2, 1]), and the exponents of the dividends whose quotient is formed here,
// lo .. lo + span - 1 (none for a b that is not a normal number).  A quotient of
// y falls short of the exact one by less than 6 2^55 2^-64 < 1, so it is the
// integer below that or the next below.
struct Recip {
    double b;
    unsigned long long y;
    int lo;
    unsigned span;
};
__device__ __forceinline__ Recip recip(double b) {
    Recip r;
    r.b = b;
    const int hi = __double2hiint(b), e = (hi >> 20) & 0x7ff;
    r.lo = max(e - 1021, 1);
    r.span = e == 0 || e == 0x7ff ? 0u : (unsigned)(min(e + 1021, 2046) - r.lo + 1);
    float h, l;
    split(hi, __double2loint(b), h, l);
    const float y0 = fminf(fmaxf(rcp_ftz(h), 0.5f), 1.f);
    const float q = fmaf(-l, y0, fmaf(-h, y0, 1.f));
    const unsigned long long y = join(y0, y0 * fmaf(q, q, q));
    // 2^62 - (mantissa 2^11) y 2^-64: the residual 1 - m y in units of 2^-62
    const unsigned long long t = __umul64hi(mantissa(b) << 11, y);
    r.y = refine(y, (int)((1ull << 62) - t), 30) - 4;
    return r;
}
// a / b
__device__ __forceinline__ double div(double a, const Recip &r) {
    const int ahi = __double2hiint(a), bhi = __double2hiint(r.b), ea = (ahi >> 20) & 0x7ff;
    const int sign = (ahi ^ bhi) & 0x80000000;
    if ((unsigned)(ea - r.lo) < r.span) {
        const unsigned long long mb = mantissa(r.b);
        unsigned long long m = mantissa(a);
        int e = ea - ((bhi >> 20) & 0x7ff) + 1022;   // of the quotient, less one
        if (m < mb) { m += m; e--; }                  // m / mb in [1, 2)
        // the integer below m 2^52 / mb or the one below that
        const unsigned long long q = __umul64hi(m + m, r.y);
        const unsigned long long rem2 = ((m << 52) - q * mb) << 1;
        const unsigned long long v =
            q + (rem2 > mb ? 1 : 0) + (rem2 > 3 * mb ? 1 : 0);   // 2^52 .. 2^53
        return __hiloint2double(((int)(v >> 32) + (e << 20)) | sign, (int)(unsigned)v);
    }
    if (r.span && is_zero(a)) return __hiloint2double(sign, 0);
    return a / r.b;
}

__device__ __forceinline__ double root(double a) {
    const int hi = __double2hiint(a), e = hi >> 20;   // negative for a < 0
    if ((unsigned)(e - 1) < 2046u) {
        const int k = (e - 1023) >> 1, odd = (e - 1023) & 1;   // a = m 4^k, m in [1, 4)
        float h, l;
        split(hi, __double2loint(a), h, l);
        if (odd) { h *= 2.f; l *= 2.f; }
        const float y0 = fminf(fmaxf(rsqrt_ftz(h), 0.5f), 1.f);
        const float p = y0 * y0, pe = fmaf(y0, y0, -p);
        const float q = fmaf(-l, p, fmaf(-h, pe, fmaf(-h, p, 1.f)));   // 1 - m y0^2
        unsigned long long z = join(y0, y0 * fmaf(q * q, 0.375f, 0.5f * q));   // 2^63 / sqrt(m)
        const unsigned long long x = mantissa(a) << odd;                       // m 2^52
        // 2^60 - m z^2: the residual 1 - m z^2 in units of 2^-60
        const unsigned long long t = __umul64hi(x << 10, __umul64hi(z, z));
        z = refine(z, (int)((1ull << 60) - t), 29) - 16;
        // the integer below sqrt(x 2^52) or the one below that
        const unsigned long long s = __umul64hi(x + x, z);
        const unsigned long long rem = (x << 52) - s * s;
        const unsigned long long v = s + (rem > s ? 1 : 0) + (rem > 3 * s + 2 ? 1 : 0);
        return __hiloint2double((int)(v >> 32) + ((k + 1022) << 20), (int)(unsigned)v);
    }
    return sqrt(a);
}

}  // namespace d64
}  // namespace swadj
