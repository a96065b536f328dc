// fp32 convolution for small layers (one image, few pixels): FFMA implicit GEMM with the reduction split over the warps of a
// CTA.
//
// With few output tiles a layer's time is the latency of its reduction loop: load a tile of operands, synchronise, multiply,
// one step after another (conv_f32.cu: 1100 clocks per 16 reduction elements when every SM has one CTA).  Here every warp of a
// CTA owns a slice of the reduction -- chunks of 16 elements warp, warp + SL, ... -- and the whole output tile: it copies its
// chunks asynchronously into a ring of its own, waits for nobody else, and the warps' partial sums are added once at the end,
// in a fixed order.  Operand rows are stored as they lie in memory (reduction index contiguous, 80-byte pitch): a thread
// takes four reduction elements of its 8 pixels and 4 layers with twelve 16-byte reads, free of bank conflicts, for 128
// multiply-adds.  Layers with 16-byte pieces and tiles of 32 layers or more do the same on the matrix
// instructions where that is faster (further down).  Two layers that read the same input (the expands of a fire layer) go out as one grid.
#include <cmath>
#include <cstring>
#include <type_traits>

#include "f32_common.cuh"
#include "smem_attr.h"
#include "sqn_internal.h"
#include "tc_common.cuh"
#include "tc_host.h"

namespace sqn {
namespace {

constexpr int SK = 16;                  // reduction elements per chunk
constexpr int SPITCH = SK + 4;          // floats per operand row: rows of consecutive threads fall into different banks

struct F32SmallParams {
    const float* in;
    const float* w;
    const float* bias;
    float* out;
    int* status;
    int Cin, H, W, Cout, K, S, pad, OW, OHW, M, Kdim;
    int out_c_offset, out_c_total, relu;
    FastDiv div_ohw, div_ow, div_cin, div_k;
    int chunks;
    int n_tiles, blocks;
    int vec_store, early;
};

// TY x TX threads of a warp, RM x 4 outputs each: tiles of RM*TY pixels x 4*TX layers.
template <int TY, int RM, int SL, int ST, bool VEC>
__device__ __forceinline__ void conv_f32_small_body(const F32SmallParams& p, const int bid)
{
    constexpr int TX = 32 / TY, TM = RM * TY, TN = 4 * TX, ROWS = TM + TN;
    constexpr int SLOT = ROWS * SPITCH;                         // floats per ring slot
    extern __shared__ __align__(16) float sm_small[];
    __shared__ int3 rows[VEC ? 1 : TM];                         // scalar path: {offset, first row, first column} of every pixel's window
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int ty = lane / TX, tx = lane % TX;
    const int mt = bid / p.n_tiles, n0 = (bid - mt * p.n_tiles) * TN, m0 = mt * TM;
    float* ring = sm_small + warp * (ST * SLOT);
    const uint32_t ring_s = (uint32_t)__cvta_generic_to_shared(ring);

    auto window = [&](int m, int& off, int& ih, int& iw) {      // window of output pixel m
        if (m < p.M) {
            const int img = fast_div(m, p.div_ohw), r = m - img * p.OHW;
            const int oh = fast_div(r, p.div_ow), ow = r - oh * p.OW;
            ih = oh * p.S - p.pad; iw = ow * p.S - p.pad;
            off = ((img * p.H + ih) * p.W + iw) * p.Cin;
        } else { off = 0; ih = -(1 << 30); iw = 0; }
    };
    constexpr int NA = VEC ? TM / 8 : 1;
    int a_off[NA], a_ih[NA], a_iw[NA];
    if (VEC) {
#pragma unroll
        for (int j = 0; j < NA; ++j) window(m0 + (lane >> 2) + 8 * j, a_off[j], a_ih[j], a_iw[j]);
    } else {
        for (int r = tid; r < TM; r += 32 * SL) {
            int3 v;
            window(m0 + r, v.x, v.y, v.z);
            rows[r] = v;
        }
        __syncthreads();
    }
    // one chunk of the reduction into ring slot `slot`: pixels and kernels apart, so that kernels may be asked for early
    auto load_w = [&](int ch, int slot) {
        const uint32_t dst = ring_s + (uint32_t)(slot * SLOT + TM * SPITCH) * 4u;
        if (VEC) {
            const int k = ch * SK + 4 * (lane & 3);
#pragma unroll
            for (int j = 0; j < TN / 8; ++j) {
                const int r = (lane >> 2) + 8 * j;
                const bool ok = k < p.Kdim && n0 + r < p.Cout;
                cp_async_16(dst + (uint32_t)(r * SPITCH + 4 * (lane & 3)) * 4u, ok ? p.w + (size_t)(n0 + r) * p.Kdim + k : p.w, ok);
            }
        } else {
            const int k = ch * SK + (lane & 15);
#pragma unroll
            for (int j = 0; j < TN / 2; ++j) {
                const int r = (lane >> 4) + 2 * j;
                const bool ok = k < p.Kdim && n0 + r < p.Cout;
                cp_async_4(dst + (uint32_t)(r * SPITCH + (lane & 15)) * 4u, ok ? p.w + (size_t)(n0 + r) * p.Kdim + k : p.w, ok);
            }
        }
    };
    auto load_x = [&](int ch, int slot) {
        const uint32_t dst = ring_s + (uint32_t)(slot * SLOT) * 4u;
        const int k = ch * SK + (VEC ? 4 * (lane & 3) : lane & 15);
        const int t = fast_div(k, p.div_cin), c = k - t * p.Cin, kh = fast_div(t, p.div_k), kw = t - kh * p.K;
        const int off = (kh * p.W + kw) * p.Cin + c;
        if (VEC) {
#pragma unroll
            for (int j = 0; j < NA; ++j) {
                const bool ok = k < p.Kdim && (unsigned)(a_ih[j] + kh) < (unsigned)p.H && (unsigned)(a_iw[j] + kw) < (unsigned)p.W;
                cp_async_16(dst + (uint32_t)(((lane >> 2) + 8 * j) * SPITCH + 4 * (lane & 3)) * 4u, ok ? p.in + (a_off[j] + off) : p.in, ok);
            }
        } else {
#pragma unroll 8
            for (int j = 0; j < TM / 2; ++j) {
                const int r = (lane >> 4) + 2 * j;
                const int3 v = rows[r];
                const bool ok = k < p.Kdim && (unsigned)(v.y + kh) < (unsigned)p.H && (unsigned)(v.z + kw) < (unsigned)p.W;
                cp_async_4(dst + (uint32_t)(r * SPITCH + (lane & 15)) * 4u, ok ? p.in + (v.x + off) : p.in, ok);
            }
        }
    };

    const int mine = p.chunks > warp ? (p.chunks - warp + SL - 1) / SL : 0;
    // the first chunks' kernels may be fetched before the grid ahead has finished (a net's own parameters)
    if (!p.early) chain_wait();
#pragma unroll
    for (int i = 0; i < ST - 1; ++i)
        if (i < mine) load_w(warp + SL * i, i);
    if (p.early) chain_wait();
#pragma unroll
    for (int i = 0; i < ST - 1; ++i) {
        if (i < mine) load_x(warp + SL * i, i);
        cp_async_commit();
    }
    float acc[RM][4];
#pragma unroll
    for (int i = 0; i < RM; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) acc[i][j] = 0.f;
    for (int i = 0, slot = 0; i < mine; ++i) {
        cp_async_wait<ST - 2>();
        __syncwarp();                   // chunk i is here for every lane, and every lane has done with chunk i - 1's slot
        {
            const int nx = i + ST - 1;
            const int ns = slot == 0 ? ST - 1 : slot - 1;
            if (nx < mine) { load_w(warp + SL * nx, ns); load_x(warp + SL * nx, ns); }
            cp_async_commit();
        }
        const float* xs = ring + slot * SLOT + ty * SPITCH;
        const float* ws = ring + slot * SLOT + (TM + tx) * SPITCH;
#pragma unroll
        for (int kk = 0; kk < SK; kk += 4) {
            float4 a[RM], b[4];
#pragma unroll
            for (int r = 0; r < RM; ++r) a[r] = *reinterpret_cast<const float4*>(xs + r * TY * SPITCH + kk);
#pragma unroll
            for (int c = 0; c < 4; ++c) b[c] = *reinterpret_cast<const float4*>(ws + c * TX * SPITCH + kk);
#pragma unroll
            for (int r = 0; r < RM; ++r)
#pragma unroll
                for (int c = 0; c < 4; ++c) {
                    acc[r][c] = fmaf(a[r].x, b[c].x, acc[r][c]);
                    acc[r][c] = fmaf(a[r].y, b[c].y, acc[r][c]);
                    acc[r][c] = fmaf(a[r].z, b[c].z, acc[r][c]);
                    acc[r][c] = fmaf(a[r].w, b[c].w, acc[r][c]);
                }
        }
        if (++slot == ST) slot = 0;
    }
    cp_async_wait<0>();
    __syncwarp();
    // partial sums into the warp's own ring, then all warps' sums in order
    constexpr int RP = TN + 4;
    static_assert(TM * RP <= ST * SLOT, "the partial sums fit the ring");
#pragma unroll
    for (int r = 0; r < RM; ++r)
#pragma unroll
        for (int c = 0; c < 4; ++c) ring[(ty + TY * r) * RP + tx + TX * c] = acc[r][c];
    __syncthreads();
#pragma unroll
    for (int i0 = 0; i0 < TM * TN / 4; i0 += 32 * SL) {
        const int i = tid + i0;
        if (i >= TM * TN / 4) break;
        const int r = i / (TN / 4), l4 = 4 * (i % (TN / 4));
        const int m = m0 + r, n = n0 + l4;
        if (m >= p.M || n >= p.Cout) continue;
        float4 v = *reinterpret_cast<const float4*>(sm_small + r * RP + l4);
#pragma unroll
        for (int s = 1; s < SL; ++s) {
            const float4 q = *reinterpret_cast<const float4*>(sm_small + s * (ST * SLOT) + r * RP + l4);
            v.x += q.x; v.y += q.y; v.z += q.z; v.w += q.w;
        }
        const float* bias = p.bias + n;
        v.x += __ldg(bias);
        if (n + 1 < p.Cout) v.y += __ldg(bias + 1);
        if (n + 2 < p.Cout) v.z += __ldg(bias + 2);
        if (n + 3 < p.Cout) v.w += __ldg(bias + 3);
        if (p.relu) { v.x = fmaxf(v.x, 0.f); v.y = fmaxf(v.y, 0.f); v.z = fmaxf(v.z, 0.f); v.w = fmaxf(v.w, 0.f); }
        if (!sqn_dbg_ok(m >= 0 && p.out_c_offset + n < p.out_c_total, p.status)) continue;
        float* dst = p.out + (size_t)m * p.out_c_total + p.out_c_offset + n;
        if (p.vec_store && n + 4 <= p.Cout) *reinterpret_cast<float4*>(dst) = v;
        else {
            dst[0] = v.x;
            if (n + 1 < p.Cout) dst[1] = v.y;
            if (n + 2 < p.Cout) dst[2] = v.z;
            if (n + 3 < p.Cout) dst[3] = v.w;
        }
    }
}

__device__ __forceinline__ float4 ld_shared_f4(uint32_t a)
{
    float4 v;
    asm volatile("ld.shared.v4.f32 {%0, %1, %2, %3}, [%4];" : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w) : "r"(a) : "memory");
    return v;
}
__device__ __forceinline__ float ld_shared_f1(uint32_t a)
{
    float v;
    asm volatile("ld.shared.f32 %0, [%1];" : "=f"(v) : "r"(a) : "memory");
    return v;
}
// The same layer on the warp-level matrix instructions at fp32 precision: every operand as three bf16 numbers (split_pair), six
// of the nine products (see conv_f32_tc.cu), w0*x0 of 16 reduction elements at a time, added up in registers with rounded
// additions.  Tiles of 16*MF pixels x 8*NF layers; chunks of 16 reduction elements lie in shared memory as in global memory,
// rows of 64 bytes.  The order of a chunk's elements in the MMA's reduction is free: lane t of four takes elements 4t .. 4t+3 of
// its rows with one 16-byte read, free of bank conflicts.  A chunk of a 32 x 32 tile is 48 MMAs of 8 clocks per scheduler against 512
// multiply-adds of 1.45 and six times the reads; what bounds it is the chain of a chunk (read, split, products) in every warp.
// Multiply-adds against this kernel, one image: fire8's expand-3x3 12.2 -> 10.5 us, fire9's 6.8 -> 5.0, fire8's squeeze 5.3 -> 4.1,
// conv10 11.4 -> 9.4; 256 -> 256 3x3 at 14 x 14, 3 images: 42.0 -> 34.1.  Which layers take it: variant_of.  Error of a layer against 64 bits 0.5e-7 to 1.4e-7 (0.7e-7 to
// 4.0e-7); of outputs with a single product that is not zero 2.8e-8 (2.5e-8), with two 3.8e-8 (3.6e-8): with eight products instead of
// six 2.55e-8 and 3.6e-8, but fire4's pair 14.2 -> 15.9 us, conv10 9.5 -> 10.9.
// A tile with a sum that is not finite is computed again with multiply-adds.
template <int MF, int NF, int SL, int ST>
__device__ __forceinline__ void conv_f32_small_tc_body(const F32SmallParams& p, const int bid)
{
    constexpr int TM = 16 * MF, TN = 8 * NF, SLOT = (TM + TN) * SK * 4;      // (bytes of a ring slot)
    extern __shared__ __align__(16) float sm_small[];
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int mt = bid / p.n_tiles, n0 = (bid - mt * p.n_tiles) * TN, m0 = mt * TM;
    const uint32_t ring = (uint32_t)__cvta_generic_to_shared(sm_small) + (uint32_t)(warp * ST * SLOT);

    // this lane's copies: piece q (4 reduction elements) of rows r0 + 8 * j
    const int q = lane & 3, r0 = lane >> 2;
    __shared__ int4 rows[TM];                   // {offset, first row, first column} of every pixel's window
    if (tid < TM) {
        const int m = m0 + tid;
        int4 v = make_int4(0, -(1 << 30), 0, 0);
        if (m < p.M) {
            const int img = fast_div(m, p.div_ohw), r = m - img * p.OHW;
            const int oh = fast_div(r, p.div_ow), ow = r - oh * p.OW;
            v.y = oh * p.S - p.pad; v.z = ow * p.S - p.pad;
            v.x = ((img * p.H + v.y) * p.W + v.z) * p.Cin;
        }
        rows[tid] = v;
    }
    __syncthreads();
    const uint32_t my_piece = (uint32_t)(16 * lane);
    auto load_w = [&](int ch, int slot) {
        const uint32_t dst = ring + (uint32_t)(slot * SLOT + TM * SK * 4) + my_piece;
        const int k = ch * SK + 4 * q;
#pragma unroll
        for (int j = 0; j < NF; ++j) {
            const bool ok = k < p.Kdim && n0 + r0 + 8 * j < p.Cout;
            cp_async_16(dst + (uint32_t)(512 * j), ok ? p.w + (size_t)(n0 + r0 + 8 * j) * p.Kdim + k : p.w, ok);
        }
    };
    auto load_x = [&](int ch, int slot) {
        const uint32_t dst = ring + (uint32_t)(slot * SLOT) + my_piece;
        const int k = ch * SK + 4 * q;
        const int t = fast_div(k, p.div_cin), c = k - t * p.Cin, kh = fast_div(t, p.div_k), kw = t - kh * p.K;
        const int off = (kh * p.W + kw) * p.Cin + c;
#pragma unroll
        for (int j = 0; j < 2 * MF; ++j) {
            const int4 v = rows[r0 + 8 * j];
            const bool ok = k < p.Kdim && (unsigned)(v.y + kh) < (unsigned)p.H && (unsigned)(v.z + kw) < (unsigned)p.W;
            cp_async_16(dst + (uint32_t)(512 * j), ok ? p.in + (v.x + off) : p.in, ok);
        }
    };
    const int mine = p.chunks > warp ? (p.chunks - warp + SL - 1) / SL : 0;
    const int g = lane >> 2, t4 = lane & 3;
    const uint32_t xr = ring + (uint32_t)(g * 64 + t4 * 16), wr = xr + (uint32_t)(TM * 64);
    constexpr int RP = TN + 4;
    static_assert(TM * RP * 4 <= ST * SLOT, "the partial sums fit the ring");
    // the first chunks' kernels may be fetched before the grid ahead has finished (a net's own parameters)
    if (!p.early) chain_wait();
    for (bool exact = false;; exact = true) {
#pragma unroll
        for (int i = 0; i < ST - 1; ++i)
            if (i < mine) load_w(warp + SL * i, i);
        if (p.early && !exact) chain_wait();
#pragma unroll
        for (int i = 0; i < ST - 1; ++i) {
            if (i < mine) load_x(warp + SL * i, i);
            cp_async_commit();
        }
        float acc[NF][MF][4];
#pragma unroll
        for (int f = 0; f < NF; ++f)
#pragma unroll
            for (int e = 0; e < MF; ++e)
#pragma unroll
                for (int i = 0; i < 4; ++i) acc[f][e][i] = 0.f;
        for (int i = 0, slot = 0; i < mine; ++i) {
            cp_async_wait<ST - 2>();
            __syncwarp();               // chunk i is here for every lane, and every lane has done with chunk i - 1's slot
            {
                const int nx = i + ST - 1, ns = slot == 0 ? ST - 1 : slot - 1;
                if (nx < mine) { load_w(warp + SL * nx, ns); load_x(warp + SL * nx, ns); }
                cp_async_commit();
            }
            const uint32_t xs = xr + (uint32_t)(slot * SLOT), ws = wr + (uint32_t)(slot * SLOT);
            if (!exact) {
                uint32_t xh[MF][4], xm[MF][4], xl[MF][4];
#pragma unroll
                for (int e = 0; e < MF; ++e)
#pragma unroll
                    for (int h = 0; h < 2; ++h) {           // rows g and g + 8
                        const float4 v = ld_shared_f4(xs + (uint32_t)((16 * e + 8 * h) * 64));
                        split_pair(v.x, v.y, xh[e][h], xm[e][h], xl[e][h]);
                        split_pair(v.z, v.w, xh[e][2 + h], xm[e][2 + h], xl[e][2 + h]);
                    }
                auto layers = [&](auto count, int f0) {     // tiles of 8 layers f0 ..
                    constexpr int F = decltype(count)::value;
                    uint32_t wh[F][2], wm[F][2], wl[F][2];
#pragma unroll
                    for (int f = 0; f < F; ++f) {
                        const float4 v = ld_shared_f4(ws + (uint32_t)(8 * (f0 + f) * 64));
                        split_pair(v.x, v.y, wh[f][0], wm[f][0], wl[f][0]);
                        split_pair(v.z, v.w, wh[f][1], wm[f][1], wl[f][1]);
                    }
                    mma_split(&acc[f0], xh, xm, xl, wh, wm, wl);
                };
#pragma unroll
                for (int f = 0; f + 2 <= NF; f += 2) layers(std::integral_constant<int, 2>(), f);
                if (NF % 2) layers(std::integral_constant<int, 1>(), NF - 1);
            } else {
                const uint32_t x0 = xs - (uint32_t)(t4 * 16), w0 = ws - (uint32_t)(t4 * 16 + g * 64) + (uint32_t)(2 * t4 * 64);
#pragma unroll 1
                for (int k = 0; k < SK; ++k) {
                    float w[NF][2];
#pragma unroll
                    for (int f = 0; f < NF; ++f) { w[f][0] = ld_shared_f1(w0 + 4u * k + (uint32_t)(8 * f * 64)); w[f][1] = ld_shared_f1(w0 + 4u * k + (uint32_t)(8 * f * 64 + 64)); }
#pragma unroll
                    for (int e = 0; e < MF; ++e) {
                        const float xa = ld_shared_f1(x0 + 4u * k + (uint32_t)(16 * e * 64)), xb = ld_shared_f1(x0 + 4u * k + (uint32_t)((16 * e + 8) * 64));
#pragma unroll
                        for (int f = 0; f < NF; ++f) {
                            acc[f][e][0] = fmaf(xa, w[f][0], acc[f][e][0]); acc[f][e][1] = fmaf(xa, w[f][1], acc[f][e][1]);
                            acc[f][e][2] = fmaf(xb, w[f][0], acc[f][e][2]); acc[f][e][3] = fmaf(xb, w[f][1], acc[f][e][3]);
                        }
                    }
                }
            }
            if (++slot == ST) slot = 0;
        }
        cp_async_wait<0>();
        __syncwarp();
        // partial sums into the warp's own ring, then all warps' sums in order
        float* part = sm_small + warp * (ST * SLOT / 4);
#pragma unroll
        for (int e = 0; e < MF; ++e)
#pragma unroll
            for (int f = 0; f < NF; ++f) {
                float* d = part + (16 * e + g) * RP + 8 * f + 2 * t4;
                *reinterpret_cast<float2*>(d) = make_float2(acc[f][e][0], acc[f][e][1]);
                *reinterpret_cast<float2*>(d + 8 * RP) = make_float2(acc[f][e][2], acc[f][e][3]);
            }
        __syncthreads();
        const float unscale = exact ? 1.f : SPLIT_UNSCALE;
        bool finite = true;
#pragma unroll
        for (int i0 = 0; i0 < TM * TN / 4; i0 += 32 * SL) {
            const int i = tid + i0;
            if (i >= TM * TN / 4) break;
            const int r = i / (TN / 4), l4 = 4 * (i % (TN / 4));
            const int m = m0 + r, n = n0 + l4;
            if (m >= p.M || n >= p.Cout) continue;
            float4 v = *reinterpret_cast<const float4*>(sm_small + r * RP + l4);
#pragma unroll
            for (int s = 1; s < SL; ++s) {
                const float4 u = *reinterpret_cast<const float4*>(sm_small + s * (ST * SLOT / 4) + r * RP + l4);
                v.x += u.x; v.y += u.y; v.z += u.z; v.w += u.w;
            }
            finite = finite && fabsf(v.x) < INFINITY && fabsf(v.y) < INFINITY && fabsf(v.z) < INFINITY && fabsf(v.w) < INFINITY;
            const float* bias = p.bias + n;
            v.x = fmaf(v.x, unscale, __ldg(bias));
            if (n + 1 < p.Cout) v.y = fmaf(v.y, unscale, __ldg(bias + 1));
            if (n + 2 < p.Cout) v.z = fmaf(v.z, unscale, __ldg(bias + 2));
            if (n + 3 < p.Cout) v.w = fmaf(v.w, unscale, __ldg(bias + 3));
            if (p.relu) { v.x = fmaxf(v.x, 0.f); v.y = fmaxf(v.y, 0.f); v.z = fmaxf(v.z, 0.f); v.w = fmaxf(v.w, 0.f); }
            if (!sqn_dbg_ok(m >= 0 && p.out_c_offset + n < p.out_c_total, p.status)) continue;
            float* dst = p.out + (size_t)m * p.out_c_total + p.out_c_offset + n;
            if (p.vec_store && n + 4 <= p.Cout) *reinterpret_cast<float4*>(dst) = v;
            else {
                dst[0] = v.x;
                if (n + 1 < p.Cout) dst[1] = v.y;
                if (n + 2 < p.Cout) dst[2] = v.z;
                if (n + 3 < p.Cout) dst[3] = v.w;
            }
        }
        if (exact || !__syncthreads_or(!finite)) break;     // (the rings are free again)
    }
}

template <int MF, int NF, int SL, int ST>
__global__ void __launch_bounds__(32 * SL, 16 / SL)
conv_f32_small_tc_kernel(const __grid_constant__ F32SmallParams p0, const __grid_constant__ F32SmallParams p1)
{
    chain_release();
    if ((int)blockIdx.x < p0.blocks) conv_f32_small_tc_body<MF, NF, SL, ST>(p0, (int)blockIdx.x);
    else conv_f32_small_tc_body<MF, NF, SL, ST>(p1, (int)blockIdx.x - p0.blocks);
}

template <int TY, int RM, int SL, int ST, bool VEC>
__global__ void __launch_bounds__(32 * SL, 16 / SL)
conv_f32_small_kernel(const __grid_constant__ F32SmallParams p0, const __grid_constant__ F32SmallParams p1)
{
    chain_release();
    if ((int)blockIdx.x < p0.blocks) conv_f32_small_body<TY, RM, SL, ST, VEC>(p0, (int)blockIdx.x);
    else conv_f32_small_body<TY, RM, SL, ST, VEC>(p1, (int)blockIdx.x - p0.blocks);
}

bool fill(const ConvDesc& d, int tm, int tn, F32SmallParams* p)
{
    std::memset(p, 0, sizeof(*p));
    const long long M = (long long)d.N * d.OH * d.OW, Kdim = (long long)d.K * d.K * d.Cin;
    if (M > 0x7fffffffLL - 512 || Kdim > 0x7fffffffLL - 64 || (long long)d.N * d.H * d.W * d.Cin > 0x3fffffffLL) return false;
    if (((long long)d.K * d.W + d.K) * d.Cin + (long long)d.pad * (d.W + 1) * d.Cin > 0x3fffffffLL) return false;
    p->in = static_cast<const float*>(d.in); p->w = static_cast<const float*>(d.w); p->bias = d.bias;
    p->out = static_cast<float*>(d.out); p->status = device_status_word();
    p->Cin = d.Cin; p->H = d.H; p->W = d.W; p->Cout = d.Cout; p->K = d.K; p->S = d.S; p->pad = d.pad;
    p->OW = d.OW; p->OHW = d.OH * d.OW; p->M = (int)M; p->Kdim = (int)Kdim;
    p->out_c_offset = d.out_c_offset; p->out_c_total = d.out_c_total; p->relu = d.relu;
    p->div_ohw = make_div(p->OHW); p->div_ow = make_div(p->OW); p->div_cin = make_div(p->Cin); p->div_k = make_div(p->K);
    p->chunks = (p->Kdim + SK - 1) / SK;
    p->n_tiles = (d.Cout + tn - 1) / tn;
    const long long blocks = ((M + tm - 1) / tm) * p->n_tiles;
    if (blocks > 0x3fffffffLL) return false;
    p->blocks = (int)blocks;
    p->vec_store = d.out_c_offset % 4 == 0 && d.out_c_total % 4 == 0;
    p->early = d.params_static;
    return true;
}

// 16-byte pieces: on the matrix instructions
template <int MF, int NF, int SL, int ST>
cudaError_t launch_tc(const F32SmallParams& a, const F32SmallParams& b, cudaStream_t stream)
{
    constexpr size_t smem = (size_t)SL * ST * (16 * MF + 8 * NF) * SK * 4;
    static SmemAttr attr;
    const cudaError_t arc = attr.allow((const void*)conv_f32_small_tc_kernel<MF, NF, SL, ST>, smem);
    if (arc != cudaSuccess) return arc;
    const cudaError_t rc =
        launch_chained(conv_f32_small_tc_kernel<MF, NF, SL, ST>, dim3((unsigned)(a.blocks + b.blocks)), dim3(32 * SL), smem, stream, a, b);
    if (rc == cudaSuccess) note_launch("conv_f32_small%s %dx%d vec, %d warps, %d slots, products", b.blocks ? " x 2" : "", 16 * MF, 8 * NF, SL, ST);
    return rc;
}

template <int TY, int RM, int SL, int ST, bool VEC>
cudaError_t launch(const F32SmallParams& a, const F32SmallParams& b, cudaStream_t stream)
{
    constexpr size_t smem = (size_t)SL * ST * (RM * TY + 128 / TY) * SPITCH * 4;
    static SmemAttr attr;
    const cudaError_t arc = attr.allow((const void*)conv_f32_small_kernel<TY, RM, SL, ST, VEC>, smem);
    if (arc != cudaSuccess) return arc;
    const cudaError_t rc =
        launch_chained(conv_f32_small_kernel<TY, RM, SL, ST, VEC>, dim3((unsigned)(a.blocks + b.blocks)), dim3(32 * SL), smem, stream, a, b);
    if (rc == cudaSuccess) note_launch("conv_f32_small%s %dx%d%s, %d warps, %d slots", b.blocks ? " x 2" : "", RM * TY, 128 / TY, VEC ? " vec" : "", SL, ST);
    return rc;
}

// Tile, warps and ring for a layer (or two) of so many tiles; measured on SqueezeNet's layers at batch 1 and 4:
//  - half as many pixels per thread where the larger tiles would leave half of the SMs without a CTA (fire9's squeeze 6.9 ->
//    4.7 us, fire5's 4.2 -> 3.2);
//  - eight warps and three slots per warp where every SM gets one CTA at most, two slots where two CTAs per SM make it one
//    wave (fire8's expand-3x3 at batch 1, 184 tiles: 14.1 -> 12.5 us), else four warps and three slots.
//  - a single layer with 16-byte pieces, more than six chunks and more tiles than two per SM: tiles of 40 or 48 layers where they
//    compute an eighth less than those of 32 and then are two per SM at most (20 -> 36 5x5/2, nine images of 61 x 47, half of the
//    32-layer tiles' work for nothing: 17.8 -> 12.8 us; 50 such layers 0.81, with six chunks or fewer 1.0).  Fewer tiles of 32 run two
//    to an SM at once and are the faster ones (150 layers, the wider tiles 1.03 to 1.24; 12 -> 48 3x3/2, six images of 50 x 50, 4.7 and 5.7 us).
struct SmallConfig { bool narrow; int rm, tm, tn; };

SmallConfig config_of(const ConvDesc* d, int n, int sms)
{
    SmallConfig c;
    c.narrow = d[0].Cout <= 16 && (n == 1 || d[1].Cout <= 16);
    c.tn = c.narrow ? 16 : 32;
    c.rm = 8;
    long long blocks = 0;
    for (int i = 0; i < n; ++i)
        blocks += (((long long)d[i].N * d[i].OH * d[i].OW + (c.narrow ? 63 : 31)) / (c.narrow ? 64 : 32)) * ((d[i].Cout + c.tn - 1) / c.tn);
    if (blocks <= sms / 2) c.rm = 4;
    else if (blocks > 2 * sms && !c.narrow && n == 1 && d[0].Cin % 4 == 0 && (long long)d[0].K * d[0].K * d[0].Cin > 6 * SK)
        for (int tn = 40; tn <= 48; tn += 8) {
            const int cols = (d[0].Cout + tn - 1) / tn;
            if (cols * tn * 8LL <= (d[0].Cout + c.tn - 1) / c.tn * c.tn * 7LL && blocks / ((d[0].Cout + 31) / 32) * cols <= 2 * sms) c.tn = tn;
        }
    c.tm = (c.narrow ? 8 : 4) * c.rm;
    return c;
}

// Warps, slots and arithmetic of a launch of so many tiles (blocks) in so many columns (0: two layers), the longest of them with so many
// chunks; shared: windows that overlap at every pixel.
struct SmallVariant { int warps, slots; bool products; };

SmallVariant variant_of(const SmallConfig& c, bool vec, long long blocks, int chunks, int columns, bool shared, int sms)
{
    const bool pair = columns == 0;
    const bool deep = chunks > 2;               // (more than two warps have chunks)
    SmallVariant v = {deep && blocks <= 2 * sms ? 8 : 4, deep && blocks > sms && blocks <= 2 * sms ? 2 : 3, false};
    if (c.tn > 32) return {8, 2, true};
    if (!vec || c.narrow) return v;
    // Where the matrix instructions are the faster ones; both timed on 1200 random layers and 600 fire layers' expands (geometric
    // means, multiply-adds = 1).  A chunk on them is a longer chain for a warp (split, products, sums), so a warp needs some; but
    // rings without padding let one CTA more live on an SM.
    if (c.rm == 4)
        // CTAs on half the SMs: 7 to 11 chunks 1.0, 12 to 64 0.95, more 0.87, 4 to 6 1.04, fewer 1.10; on more of them 4 to 8 0.96, 9 to 64
        // 0.88, more 0.86, three 1.03.  Expands of 16 squeeze layers, nine chunks, 1.02, of 32 and more 0.91.
        v.products = deep && blocks <= sms && chunks > (pair ? 9 : blocks > sms / 2 ? 3 : 6);
    else if (blocks <= sms)
        // one CTA per SM: 1.03 to 1.09 at any number of chunks.  Except one column of tiles on three quarters of the SMs: 0.94 with up to 16
        // chunks (128 -> 32 1x1 at 55 x 55 3.7 -> 3.5 us; on more of them 1.01).
        v.products = columns == 1 && deep && chunks <= 16 && blocks <= sms * 3 / 4;
    else if (blocks <= 2 * sms)
        // two CTAs per SM: 5 to 16 chunks 0.90, more 0.84, fewer 1.01; expands 0.87 (16 squeeze layers 0.93)
        v.products = chunks > 4;
    else
        // Four warps: three CTAs per SM with multiply-adds, four with products.  Up to three per SM 0.92 with one column of tiles, 0.90 with
        // a few of windows that overlap, else 0.99 to 1.07; up to four 0.67 to 0.75 (one wave instead of two), more 0.8.  Of a pair half
        // the CTAs are short: up to 4 per SM 1.02, up to 4.75 1.05 (nine chunks 0.88), more 0.94 (0.85).
        v.products = pair ? blocks > (chunks > 9 ? 19 * sms / 4 : 4 * sms) : blocks > 3 * sms || (deep && (columns == 1 || (shared && columns <= 6)));
    return v;
}

template <int TY, int RM, bool VEC>
cudaError_t launch_ty(const SmallVariant& v, const F32SmallParams& a, const F32SmallParams& b, cudaStream_t stream)
{
    if constexpr (VEC && TY == 4) {
        if (v.products) {
            if constexpr (RM == 4) return launch_tc<1, 4, 8, 3>(a, b, stream);
            else return v.warps == 4 ? launch_tc<2, 4, 4, 3>(a, b, stream) : v.slots == 2 ? launch_tc<2, 4, 8, 2>(a, b, stream) : launch_tc<2, 4, 8, 3>(a, b, stream);
        }
    }
    if (v.warps == 4) return launch<TY, RM, 4, 3, VEC>(a, b, stream);
    return v.slots == 2 ? launch<TY, RM, 8, 2, VEC>(a, b, stream) : launch<TY, RM, 8, 3, VEC>(a, b, stream);
}

template <int NF>
cudaError_t launch_wide(const F32SmallParams& a, const F32SmallParams& b, cudaStream_t stream)
{
    return launch_tc<2, NF, 8, 2>(a, b, stream);
}

}  // namespace

// Microseconds: a launch, then the busiest SM's tiles by their chunks.  With 16-byte pieces: eight warps by the variant that would run, and
// the wide tiles, fitted to 640 random layers (0.88 to 1.1 of it in nine of ten); four warps by the multiply-adds' 260 clocks per chunk
// (150 with the smaller tile), of which products take two thirds to three quarters.  With the narrow tile 300 clocks per chunk, and where warps take several, as if every warp had as many
// as the one with the most: fire2's squeeze, 6 chunks for 4 warps, 12.9 us at 19 images, 16.5 at 25, 40 at 71 (FFMA 14.5, 14.5, 37),
// fire3's, 8 chunks, 14.3 at 19, 67 at 116 (FFMA 18.6, 76).  Where the operands come in pieces of 4 bytes 500 clocks (450 with the
// smaller tile, 900 with the narrow one) and more for a tile's start, fitted to 450 random layers (0.85 to 1.15 of it in eight
// of ten; 750 for all of them gave 0.46).
float f32_small_estimate(const ConvDesc& d, int sms)
{
    const SmallConfig c = config_of(&d, 1, sms);
    const int n_tiles = (d.Cout + c.tn - 1) / c.tn;
    const long long blocks = (((long long)d.N * d.OH * d.OW + c.tm - 1) / c.tm) * n_tiles, Kdim = (long long)d.K * d.K * d.Cin;
    const float chunks = (float)((Kdim + SK - 1) / SK);
    const float rounds = (float)((blocks + sms - 1) / sms);
    if (d.Cin % 4 != 0) return 2.7f + rounds * (chunks * (c.rm == 4 ? 450.f : c.narrow ? 900.f : 500.f) + 1650.f) / 1965.f;
    if (c.tn > 32) return c.tn == 40 ? 2.9f + 0.285f * chunks : 3.3f + 0.316f * chunks;         // (two CTAs per SM)
    const SmallVariant v = variant_of(c, true, blocks, Kdim < (1 << 20) ? (int)chunks : 1 << 16, n_tiles, d.K > 1 && d.S == 1, sms);
    if (!c.narrow && v.warps == 8) {
        if (c.rm == 4) return v.products ? 1.7f + 0.07f * chunks * (float)blocks / (float)sms + 0.53f * ceilf(chunks / 8.f) : 1.75f + 0.084f * chunks;
        if (v.slots == 3) return 2.2f + 0.166f * chunks;
        return v.products ? 2.55f + 0.228f * chunks : 2.65f + 0.21f * chunks;
    }
    const float warps = blocks > 2 * sms ? 4.f : 8.f;
    const float narrow = 300.f * (chunks > warps ? warps * ceilf(chunks / warps) : chunks);
    const float us = rounds * ((c.rm == 4 ? 150.f * chunks : c.narrow ? narrow : 260.f * chunks) + 450.f) / 1965.f;
    return 2.2f + (blocks > 2 * sms ? 1.2f * us : us);
}

int launch_conv_f32_small(const ConvDesc* d, int n, cudaStream_t stream)
{
    const int sms = sm_count();
    const SmallConfig c = config_of(d, n, sms);
    bool vec = true;
    F32SmallParams p[2];
    for (int i = 0; i < n; ++i) {
        if (!fill(d[i], c.tm, c.tn, &p[i])) return SQN_ERR_UNSUPPORTED;
        vec = vec && d[i].Cin % 4 == 0;
    }
    if (n == 1) { p[1] = p[0]; p[1].blocks = 0; }
    const int chunks = n == 2 && p[1].chunks > p[0].chunks ? p[1].chunks : p[0].chunks;
    const SmallVariant v = variant_of(c, vec, (long long)p[0].blocks + p[1].blocks, chunks, n == 1 ? p[0].n_tiles : 0, d[0].K > 1 && d[0].S == 1, sms);
    cudaError_t rc;
    if (c.tn > 32) rc = c.tn == 40 ? launch_wide<5>(p[0], p[1], stream) : launch_wide<6>(p[0], p[1], stream);
    else if (c.rm == 8) rc = c.narrow ? (vec ? launch_ty<8, 8, true>(v, p[0], p[1], stream) : launch_ty<8, 8, false>(v, p[0], p[1], stream))
                                 : (vec ? launch_ty<4, 8, true>(v, p[0], p[1], stream) : launch_ty<4, 8, false>(v, p[0], p[1], stream));
    else rc = c.narrow ? (vec ? launch_ty<8, 4, true>(v, p[0], p[1], stream) : launch_ty<8, 4, false>(v, p[0], p[1], stream))
                       : (vec ? launch_ty<4, 4, true>(v, p[0], p[1], stream) : launch_ty<4, 4, false>(v, p[0], p[1], stream));
    if (rc != cudaSuccess) return SQN_ERR_CUDA;
    return cudaGetLastError() == cudaSuccess ? SQN_OK : SQN_ERR_CUDA;
}

}  // namespace sqn
