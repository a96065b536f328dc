// Shared by the fp32 kernels: division by a constant and asynchronous copies.
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

}  // namespace sqn
