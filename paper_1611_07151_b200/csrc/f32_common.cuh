// Shared by the fp32 kernels: division by a constant, asynchronous copies, and the exact split of fp32 operands into bf16 numbers.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

namespace sqn {

struct FastDiv { unsigned mul; int shift; };        // n / d for 0 <= n < 2^31 (mul = 0: d = 1)
inline FastDiv make_div(int d)
{
    FastDiv f = {0u, 0};
    if (d <= 1) return f;
    int l = 0;
    while ((1ll << l) < d) ++l;
    f.mul = (unsigned)(((1ull << (31 + l)) + (unsigned)d - 1) / (unsigned)d);
    f.shift = l - 1;
    return f;
}

__device__ __forceinline__ int fast_div(int n, FastDiv d)
{
    return d.mul ? (int)(__umulhi((unsigned)n, d.mul) >> d.shift) : n;
}

__device__ __forceinline__ void cp_async_16(uint32_t dst, const void* src, bool ok)
{
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst), "l"(src), "r"(ok ? 16 : 0) : "memory");
}
__device__ __forceinline__ void cp_async_4(uint32_t dst, const void* src, bool ok)
{
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;" ::"r"(dst), "l"(src), "r"(ok ? 4 : 0) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int PENDING>
__device__ __forceinline__ void cp_async_wait() { asm volatile("cp.async.wait_group %0;" ::"n"(PENDING) : "memory"); }

// Operands are multiplied by this before they are split into three bf16 numbers: the last bit of the smallest fp32 number, 2^-149,
// is then bf16's smallest subnormal number, 2^-133, so that all three parts of any number are exact (without it a number of 1e-36
// kept 14 bits, one of 1e-40 one).  Sums carry its square.  What overflows by it (operands from 2^112, sums from 2^96) is not finite
// and computed again with multiply-adds.
constexpr float SPLIT_SCALE = 0x1p16f, SPLIT_UNSCALE = 0x1p-32f;

// Two fp32 differences (the bits of all operands), one instruction
__device__ __forceinline__ void sub2(uint32_t ax, uint32_t ay, uint32_t bx, uint32_t by, uint32_t& dx, uint32_t& dy)
{
    asm("{\n\t.reg .b64 a, b;\n\t"
        "mov.b64 a, {%2, %3};\n\t"
        "mov.b64 b, {%4, %5};\n\t"
        "sub.rn.f32x2 a, a, b;\n\t"
        "mov.b64 {%0, %1}, a;\n\t}"
        : "=r"(dx), "=r"(dy) : "r"(ax), "r"(ay), "r"(bx), "r"(by));
}
// Two values as three packed bf16 pairs whose sums are SPLIT_SCALE times the values (the split of Henry, Tang and Heinecke, "Leveraging the
// bfloat16 Artificial Intelligence Datatype For Higher-Precision Computations", 2019).  The first is the value rounded to nearest
// (the remainder is below 2^-8 of it and of either sign), the second the leading eight bits of the remainder, the third the rest.
__device__ __forceinline__ void split_pair(float x, float y, uint32_t& h, uint32_t& m, uint32_t& l)
{
    asm("{\n\t.reg .b64 a, b;\n\t"
        "mov.b64 a, {%0, %1};\n\t"
        "mov.b64 b, {%2, %2};\n\t"
        "mul.rn.f32x2 a, a, b;\n\t"
        "mov.b64 {%0, %1}, a;\n\t}"
        : "+f"(x), "+f"(y) : "f"(SPLIT_SCALE));
    asm("cvt.rn.bf16x2.f32 %0, %1, %2;" : "=r"(h) : "f"(y), "f"(x));
    uint32_t rx, ry, sx, sy;
    sub2(__float_as_uint(x), __float_as_uint(y), h << 16, h & 0xffff0000u, rx, ry);         // at most 16 significant bits
    m = __byte_perm(rx, ry, 0x7632);
    sub2(rx, ry, rx & 0xffff0000u, ry & 0xffff0000u, sx, sy);                               // at most 8
    l = __byte_perm(sx, sy, 0x7632);
}

}  // namespace sqn
