// Device helpers shared by the tensor-core kernels: the bounded mbarrier wait and the fp32 -> bf16 packing.
#pragma once

#include <cuda_bf16.h>
#include <cuda_fp16.h>

#include "ptx_sm100.cuh"
#include "sqn_internal.h"

namespace sqn {

constexpr long long WAIT_LIMIT_CYCLES = 4000000000LL;   // about two seconds

// Bounded mbarrier wait.  Polls back to back at first (hand-offs between the roles take a few
// hundred cycles), backs off with nanosleep on long waits, and gives up after `limit` cycles:
// the CTA then records SQN_ERR_TIMEOUT and every role leaves its loop.
__device__ __forceinline__ bool wait_bar_limit(uint32_t bar, uint32_t parity, volatile int* abort_flag, int* status, long long limit)
{
    if (ptx::mbar_try_wait(bar, parity)) return true;
    const long long t0 = clock64();
    for (uint32_t i = 1;; ++i) {
        if (ptx::mbar_try_wait(bar, parity)) return true;
        if ((i & 255u) == 0u) {
            if (*abort_flag) return false;
            if (clock64() - t0 > limit) {
                *abort_flag = 1;
                if (status) atomicExch(status, (int)SQN_ERR_TIMEOUT);
                return false;
            }
        }
        if (i > 4096u) __nanosleep(128);
    }
}
__device__ __forceinline__ bool wait_bar(uint32_t bar, uint32_t parity, volatile int* abort_flag, int* status)
{
    return wait_bar_limit(bar, parity, abort_flag, status, WAIT_LIMIT_CYCLES);
}

// The 16-bit storage type of the tensor-core paths is bf16, or fp16 where `f16` is set (same size, same layouts).
// two fp32 values -> packed pair, round to nearest even
__device__ __forceinline__ uint32_t pack_x2(float lo, float hi, int f16)
{
    uint32_t d;
    if (f16) asm("cvt.rn.f16x2.f32 %0, %1, %2;" : "=r"(d) : "f"(hi), "f"(lo));
    else asm("cvt.rn.bf16x2.f32 %0, %1, %2;" : "=r"(d) : "f"(hi), "f"(lo));
    return d;
}
// max(.,0) and the conversion of two values in one instruction
__device__ __forceinline__ uint32_t pack_relu_x2(float lo, float hi, int f16)
{
    uint32_t d;
    if (f16) asm("cvt.rn.relu.f16x2.f32 %0, %1, %2;" : "=r"(d) : "f"(hi), "f"(lo));
    else asm("cvt.rn.relu.bf16x2.f32 %0, %1, %2;" : "=r"(d) : "f"(hi), "f"(lo));
    return d;
}

// maximum of three values in one instruction
__device__ __forceinline__ float max3(float a, float b, float c)
{
    float r;
    asm("max.f32 %0, %1, %2, %3;" : "=f"(r) : "f"(a), "f"(b), "f"(c));
    return r;
}
// fp32 -> 16 bits (round to nearest even), with max(., 0) folded into the conversion when relu is set
__device__ __forceinline__ unsigned short to_16_bits(float v, int relu, int f16)
{
    unsigned short h;
    if (f16) {
        if (relu) asm("cvt.rn.relu.f16.f32 %0, %1;" : "=h"(h) : "f"(v));
        else asm("cvt.rn.f16.f32 %0, %1;" : "=h"(h) : "f"(v));
    } else {
        if (relu) asm("cvt.rn.relu.bf16.f32 %0, %1;" : "=h"(h) : "f"(v));
        else asm("cvt.rn.bf16.f32 %0, %1;" : "=h"(h) : "f"(v));
    }
    return h;
}
// 1.0 twice
__device__ __forceinline__ uint32_t one_x2(int f16) { return f16 ? 0x3c003c00u : 0x3f803f80u; }
// b as {hi, lo} with hi + lo = b to 16 (bf16) or 22 (fp16) bits below its leading bit
__device__ __forceinline__ uint32_t bias_hi_lo(float b, int f16)
{
    if (f16) {
        const __half hi = __float2half_rn(b);
        const __half lo = __float2half_rn(b - __half2float(hi));
        return (uint32_t)__half_as_ushort(hi) | ((uint32_t)__half_as_ushort(lo) << 16);
    }
    const __nv_bfloat16 hi = __float2bfloat16_rn(b);
    const __nv_bfloat16 lo = __float2bfloat16_rn(b - __bfloat162float(hi));
    return (uint32_t)__bfloat16_as_ushort(hi) | ((uint32_t)__bfloat16_as_ushort(lo) << 16);
}
// Bias row of the bias MMAs: one 32-byte row {hi, lo, 0, ...} per output layer in the 32-byte swizzle.
__device__ __forceinline__ void bias_row(uint4* rows, int c, float b, int f16)
{
    const int u = (c >> 2) & 1;
    rows[2 * c + u] = make_uint4(bias_hi_lo(b, f16), 0u, 0u, 0u);
    rows[2 * c + (u ^ 1)] = make_uint4(0u, 0u, 0u, 0u);
}

// Warp-level matrix instructions, for layers too small for the set-up that tcgen05 needs.
__device__ __forceinline__ void ldmatrix_x4(uint32_t (&r)[4], uint32_t addr)
{
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0, %1, %2, %3}, [%4];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(addr) : "memory");
}
template <bool F16>
__device__ __forceinline__ void mma_16816(float (&c)[4], const uint32_t (&a)[4], uint32_t b0, uint32_t b1)
{
    if (F16)
        asm volatile("mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, {%0, %1, %2, %3};"
                     : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3]) : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
    else
        asm volatile("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, {%0, %1, %2, %3};"
                     : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3]) : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}

// c += a * b for bf16 operands; free to be moved among other instructions (FIRST: c = a * b)
template <bool FIRST>
__device__ __forceinline__ void mma_bf16_free(float (&c)[4], const uint32_t (&a)[4], const uint32_t (&b)[2])
{
    if (FIRST)
        asm("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, {%10, %10, %10, %10};"
            : "=f"(c[0]), "=f"(c[1]), "=f"(c[2]), "=f"(c[3])
            : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b[0]), "r"(b[1]), "f"(0.f));
    else
        asm("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, {%0, %1, %2, %3};"
            : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3]) : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b[0]), "r"(b[1]));
}
// What the matrix instructions cut off a sum of 16 products on average, added back with the corrections: an error of one sign adds up
// from layer to layer.  It grows with the number of products that are not zero.  Mean signed error of a layer without it (20 layers of
// 256 to 576 products per output, inputs |N(0, 1)| of which a share is set to zero), kernels of both signs / of one: no zeros 1.14e-8 /
// 1.65e-8 of the output, a quarter 8.1e-9 / 1.11e-8, half 5.0e-9 / 6.2e-9, three quarters 2.0e-9 / 2.1e-9, one product 0.  This is the value
// for half, maps behind a ReLU, with kernels of both signs; dense inputs keep 6e-9 (one sign 1.1e-8) too little, few products up to
// 5e-9 too much.  The corrections have to be summed apart: with all six products in one sum 3.9e-8 were cut off.
constexpr float MMA_CUT = 5e-9f;

// a += c + (c * MMA_CUT + r) for two numbers at a time, each operation rounded to nearest
__device__ __forceinline__ void add_products2(float& a0, float& a1, float c0, float c1, float r0, float r1)
{
    asm("{\n\t.reg .b64 a, c, r, k;\n\t"
        "mov.b64 a, {%0, %1};\n\t"
        "mov.b64 c, {%2, %3};\n\t"
        "mov.b64 r, {%4, %5};\n\t"
        "mov.b64 k, {%6, %6};\n\t"
        "fma.rn.f32x2 r, c, k, r;\n\t"
        "add.rn.f32x2 r, c, r;\n\t"
        "add.rn.f32x2 a, a, r;\n\t"
        "mov.b64 {%0, %1}, a;\n\t}"
        : "+f"(a0), "+f"(a1) : "f"(c0), "f"(c1), "f"(r0), "f"(r1), "f"(MMA_CUT));
}

// One step of 16 reduction elements of fp32 products, operands split into three bf16 numbers each (f32_common.cuh), for F tiles of 8
// layers x N tiles of 16 pixels: the product of the first numbers and, summed on their own, the five next ones of the nine; both added
// to acc with rounded additions (the matrix instructions cut their sums off).  The tiles take every product in turn: an MMA's
// result is there after some 33 clocks, four of them take 32 to issue.
template <int F, int N>
__device__ __forceinline__ void mma_split(float (*acc)[N][4], const uint32_t (&xh)[N][4], const uint32_t (&xm)[N][4], const uint32_t (&xl)[N][4],
                                          const uint32_t (&wh)[F][2], const uint32_t (&wm)[F][2], const uint32_t (&wl)[F][2])
{
    float c[F][N][4], r[F][N][4];
#pragma unroll
    for (int p = 0; p < 6; ++p)
#pragma unroll
        for (int f = 0; f < F; ++f)
#pragma unroll
            for (int e = 0; e < N; ++e) {
                if (p == 0) mma_bf16_free<true>(r[f][e], xl[e], wh[f]);
                else if (p == 1) mma_bf16_free<false>(r[f][e], xm[e], wm[f]);
                else if (p == 2) mma_bf16_free<false>(r[f][e], xh[e], wl[f]);
                else if (p == 3) mma_bf16_free<true>(c[f][e], xh[e], wh[f]);
                else if (p == 4) mma_bf16_free<false>(r[f][e], xm[e], wh[f]);
                else mma_bf16_free<false>(r[f][e], xh[e], wm[f]);
            }
#pragma unroll
    for (int f = 0; f < F; ++f)
#pragma unroll
        for (int e = 0; e < N; ++e)
#pragma unroll
            for (int k = 0; k < 4; k += 2) add_products2(acc[f][e][k], acc[f][e][k + 1], c[f][e][k], c[f][e][k + 1], r[f][e][k], r[f][e][k + 1]);
}

}  // namespace sqn
