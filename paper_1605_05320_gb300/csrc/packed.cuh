// packed.cuh -- FP32 operations of the strip kernels whose rounding is fixed
// in the source: scalar ones that the compiler never fuses, and pairs of
// floats run by packed FP32x2 instructions (hand-written PTX).  A packed
// instruction occupies the FMA pipe twice but issues once, and each half
// rounds like the scalar operation.
#pragma once
#include "swadj_internal.cuh"

namespace swadj {
namespace fp {

__device__ __forceinline__ float add(float a, float b) { return __fadd_rn(a, b); }
__device__ __forceinline__ float sub(float a, float b) { return __fsub_rn(a, b); }
__device__ __forceinline__ float mul(float a, float b) { return __fmul_rn(a, b); }

// Two floats operated on by packed instructions.
struct f2 {
    float x, y;
};
__device__ __forceinline__ f2 mk(float x, float y) { f2 r; r.x = x; r.y = y; return r; }
__device__ __forceinline__ f2 dup(float x) { return mk(x, x); }
__device__ __forceinline__ f2 fma(f2 a, f2 b, f2 c) {
    f2 r;
    asm("{\n\t.reg .b64 a, b, c, d;\n\t"
        "mov.b64 a, {%2, %3};\n\tmov.b64 b, {%4, %5};\n\tmov.b64 c, {%6, %7};\n\t"
        "fma.rn.f32x2 d, a, b, c;\n\tmov.b64 {%0, %1}, d;\n\t}"
        : "=f"(r.x), "=f"(r.y)
        : "f"(a.x), "f"(a.y), "f"(b.x), "f"(b.y), "f"(c.x), "f"(c.y));
    return r;
}
__device__ __forceinline__ f2 mul(f2 a, f2 b) {
    f2 r;
    asm("{\n\t.reg .b64 a, b, d;\n\tmov.b64 a, {%2, %3};\n\tmov.b64 b, {%4, %5};\n\t"
        "mul.rn.f32x2 d, a, b;\n\tmov.b64 {%0, %1}, d;\n\t}"
        : "=f"(r.x), "=f"(r.y) : "f"(a.x), "f"(a.y), "f"(b.x), "f"(b.y));
    return r;
}
__device__ __forceinline__ f2 add(f2 a, f2 b) {
    f2 r;
    asm("{\n\t.reg .b64 a, b, d;\n\tmov.b64 a, {%2, %3};\n\tmov.b64 b, {%4, %5};\n\t"
        "add.rn.f32x2 d, a, b;\n\tmov.b64 {%0, %1}, d;\n\t}"
        : "=f"(r.x), "=f"(r.y) : "f"(a.x), "f"(a.y), "f"(b.x), "f"(b.y));
    return r;
}
__device__ __forceinline__ f2 rcp(f2 x) { return mk(rcp_ftz(x.x), rcp_ftz(x.y)); }

// min(|a|, |b|) with the product's sign
__device__ __forceinline__ float min_xorsign(float a, float b) {
    float r;
    asm("min.xorsign.abs.f32 %0, %1, %2;" : "=f"(r) : "f"(a), "f"(b));
    return r;
}

}  // namespace fp
}  // namespace swadj
