// Packed codes -> fp16 pairs, exact.
#pragma once
#include <cuda_fp16.h>
#include <stdint.h>

__device__ __forceinline__ uint32_t hmul2(uint32_t a, uint32_t b)
{
    uint32_t r;
    asm("mul.f16x2 %0, %1, %2;" : "=r"(r) : "r"(a), "r"(b));
    return r;
}
__device__ __forceinline__ uint32_t e4m3x2_to_f16x2(uint32_t two)
{
    uint32_t r;
    asm("cvt.rn.f16x2.e4m3x2 %0, %1;" : "=r"(r) : "h"((uint16_t)two));
    return r;
}
// eight E2M1 codes -> four pairs (all four bytes unpacked at once: byte by byte it takes 1.7 times as long)
__device__ __forceinline__ void e2m1x8_to_f16(uint32_t w, uint32_t* r)
{
    asm("{\n\t.reg .b8 a, b, c, d;\n\tmov.b32 {a, b, c, d}, %4;\n\tcvt.rn.f16x2.e2m1x2 %0, a;\n\tcvt.rn.f16x2.e2m1x2 %1, b;\n\t"
        "cvt.rn.f16x2.e2m1x2 %2, c;\n\tcvt.rn.f16x2.e2m1x2 %3, d;\n\t}" : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(w));
}
// Where bit `bit` of m is set: sixteen E4M3 codes -> eight pairs; else the pairs stay
__device__ __forceinline__ void e4m3x16_to_f16_if(uint32_t m, uint32_t bit, uint32_t w0, uint32_t w1, uint32_t w2, uint32_t w3, uint32_t* r)
{
    asm("{\n\t.reg .pred p;\n\t.reg .b32 t;\n\t.reg .b16 a, b, c, d, e, f, g, h;\n\tand.b32 t, %12, %13;\n\tsetp.ne.u32 p, t, 0;\n\t"
        "mov.b32 {a, b}, %8;\n\tmov.b32 {c, d}, %9;\n\tmov.b32 {e, f}, %10;\n\tmov.b32 {g, h}, %11;\n\t"
        "@p cvt.rn.f16x2.e4m3x2 %0, a;\n\t@p cvt.rn.f16x2.e4m3x2 %1, b;\n\t@p cvt.rn.f16x2.e4m3x2 %2, c;\n\t@p cvt.rn.f16x2.e4m3x2 %3, d;\n\t"
        "@p cvt.rn.f16x2.e4m3x2 %4, e;\n\t@p cvt.rn.f16x2.e4m3x2 %5, f;\n\t@p cvt.rn.f16x2.e4m3x2 %6, g;\n\t@p cvt.rn.f16x2.e4m3x2 %7, h;\n\t}"
        : "+r"(r[0]), "+r"(r[1]), "+r"(r[2]), "+r"(r[3]), "+r"(r[4]), "+r"(r[5]), "+r"(r[6]), "+r"(r[7])
        : "r"(w0), "r"(w1), "r"(w2), "r"(w3), "r"(m), "r"(bit));
}
// Where bit `bit` of m is set: eight bytes of shared memory from hs, which moves on behind them, and the factor; else all stay
__device__ __forceinline__ void fp8_half(uint32_t m, uint32_t bit, uint32_t& hs, uint2& hi, uint32_t& d, uint32_t factor)
{
    asm volatile("{\n\t.reg .pred p;\n\t.reg .b32 t;\n\tand.b32 t, %4, %5;\n\tsetp.ne.u32 p, t, 0;\n\t@p ld.shared.v2.b32 {%1, %2}, [%0];\n\t"
                 "@p add.u32 %0, %0, 8;\n\t@p mov.b32 %3, %6;\n\t}"
                 : "+r"(hs), "=r"(hi.x), "=r"(hi.y), "+r"(d) : "r"(m), "r"(bit), "r"(factor));
}
