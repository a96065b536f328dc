// The fp32 stem (7x7/2 on 3 layers, 96 output layers) and the 3x3/2 max-pool behind it for one image, in one launch that stores both
// maps.
//
// At one image the stem is latency, not work: as two launches, convolution on the tensor cores (its 96 tiles leave a third of the
// SMs without one) and pool, it took 17 and 5 us of a forward's 146.  Here a CTA takes 4 x 6 pooled pixels, i.e. 9 x 13 = 117
// convolution pixels (140 CTAs for 227 x 227: one wave), a warp 32 pixels x 48 layers of them on the warp-level matrix instructions at
// fp32 precision (see conv_f32_small.cu).  Kernels and the input patch lie in shared memory as in global memory; lane t of four takes
// the reduction elements 4t .. 4t+3 of every 16, those of a pixel's window by a table of offsets.  The matrix instructions bound
// it: 10 blocks of 16 reduction elements, 72 MMAs of 8 clocks per scheduler and warp each, are 6 us.
// Sums that are not finite are computed again with multiply-adds, those alone: a pixel that two tiles compute has one value.
#include <cstring>

#include "f32_common.cuh"
#include "smem_attr.h"
#include "sqn_internal.h"
#include "tc_common.cuh"
#include "tc_host.h"

namespace sqn {
namespace {

constexpr int FO = 96, FK = 147, FKB = 10;      // output layers, reduction elements, blocks of 16 of them
constexpr int FPH = 4, FPW = 6;                 // pooled pixels of a CTA
constexpr int FCH = 2 * FPH + 1, FCW = 2 * FPW + 1, FPIX = FCH * FCW;       // convolution pixels (117 of 8 x 16)
constexpr int FXH = 2 * FCH + 5, FXN = 3 * (2 * FCW + 5), FXP = 96;         // input rows, floats per input row, their pitch
constexpr int FWP = 176;                        // floats per kernel row: rows of consecutive lanes 16 banks apart
constexpr int FYP = 100;                        // floats per convolution pixel
constexpr int F_OFF_X = FO * FWP, F_OFF_Y = F_OFF_X + FXH * FXP, F_OFF_T = F_OFF_Y + 128 * FYP;
constexpr size_t F_SMEM = (size_t)(F_OFF_T + 16 * FKB) * 4;
static_assert(FPIX <= 128 && FXN <= FXP && FK <= 16 * FKB, "");

struct StemF32Params {
    const float* in;            // [N][H][W][3]
    const float* w;             // [96][7][7][3]
    const float* bias;
    float4* conv;               // [N][OH][OW][96]
    float4* pool;               // [N][PH][PW][96]
    int* status;
    int H, W, OH, OW, PH, PW, tiles_x, tiles;       // tiles per image
    int early;                  // the kernels are not written by the grid ahead
};

__device__ __forceinline__ float4 max4(float4 a, float4 b)
{
    return make_float4(fmaxf(a.x, b.x), fmaxf(a.y, b.y), fmaxf(a.z, b.z), fmaxf(a.w, b.w));
}

__global__ void __launch_bounds__(256) stem_small_f32_kernel(const __grid_constant__ StemF32Params p)
{
    extern __shared__ __align__(16) float sm_stem_f32[];
    float *sw = sm_stem_f32, *sx = sm_stem_f32 + F_OFF_X, *sy = sm_stem_f32 + F_OFF_Y;
    int* tbl = reinterpret_cast<int*>(sm_stem_f32 + F_OFF_T);       // reduction element -> float of the window
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int img = (int)blockIdx.x / p.tiles, tile = (int)blockIdx.x - img * p.tiles;
    const int ty = tile / p.tiles_x, tx = tile - ty * p.tiles_x;
    const int cy0 = 2 * FPH * ty, cx0 = 2 * FPW * tx;               // first convolution pixel; the input patch starts at twice that
    chain_release();
    if (tid < 16 * FKB) tbl[tid] = tid < FK ? tid / 21 * FXP + tid % 21 : 0;
    if (!p.early) chain_wait();
#pragma unroll 7
    for (int i = tid; i < FO * FK / 4; i += 256) {
        const float4 v = __ldg(reinterpret_cast<const float4*>(p.w) + i);
        const float e[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const int m = (4 * i + j) / FK;
            sw[m * FWP + 4 * i + j - m * FK] = e[j];
        }
    }
    for (int i = tid; i < FO * (16 * FKB - FK); i += 256) {
        const int m = i / (16 * FKB - FK);
        sw[m * FWP + FK + i - m * (16 * FKB - FK)] = 0.f;
    }
    if (p.early) chain_wait();
    {
        const float* in = p.in + (size_t)img * p.H * p.W * 3;
#pragma unroll 3
        for (int i = tid; i < FXH * FXP; i += 256) {
            const int y = i / FXP, x = i - y * FXP, iy = 2 * cy0 + y, ix = 6 * cx0 + x;
            sx[i] = iy < p.H && ix < 3 * p.W ? __ldg(in + iy * (3 * p.W) + ix) : 0.f;
        }
    }
    __syncthreads();

    // a warp: 32 pixels x 48 layers
    const int mg = warp >> 1, nh = warp & 1, g = lane >> 2, t4 = lane & 3;
    const float* win[2][2];                     // windows of this lane's pixels
#pragma unroll
    for (int e = 0; e < 2; ++e)
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            int m = 32 * mg + 16 * e + 8 * h + g;
            if (m >= FPIX) m = 0;               // (rows past the tile: computed and dropped)
            const int r = m / FCW, c = m - FCW * r;
            win[e][h] = sx + 2 * r * FXP + 6 * c;
        }
    float acc[6][2][4];
    bool finite = true;
    auto store = [&](float unscale, bool again) {       // bias and ReLU, the convolution's pixels side by side; NaN: to be computed again
#pragma unroll
        for (int j = 0; j < 6; ++j) {
            const int n = 48 * nh + 8 * j + 2 * t4;
            const float2 b = __ldg(reinterpret_cast<const float2*>(p.bias + n));
#pragma unroll
            for (int e = 0; e < 2; ++e)
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    const float s0 = acc[j][e][2 * h], s1 = acc[j][e][2 * h + 1];
                    float2* dst = reinterpret_cast<float2*>(sy + (32 * mg + 16 * e + 8 * h + g) * FYP + n);
                    float2 v = make_float2(fmaxf(fmaf(s0, unscale, b.x), 0.f), fmaxf(fmaf(s1, unscale, b.y), 0.f));     // (never NaN)
                    if (again) {
                        const float2 old = *dst;
                        if (old.x == old.x) v.x = old.x;
                        if (old.y == old.y) v.y = old.y;
                    } else {
                        if (!(fabsf(s0) < INFINITY)) { v.x = NAN; finite = false; }
                        if (!(fabsf(s1) < INFINITY)) { v.y = NAN; finite = false; }
                    }
                    *dst = v;
                }
        }
    };
#pragma unroll
    for (int e = 0; e < 2; ++e)
#pragma unroll
        for (int j = 0; j < 6; ++j)
#pragma unroll
            for (int i = 0; i < 4; ++i) acc[j][e][i] = 0.f;
    const float* wr = sw + (48 * nh + g) * FWP + 4 * t4;
#pragma unroll 1
    for (int k = 0; k < FKB; ++k) {
        const int4 o = *reinterpret_cast<const int4*>(tbl + 16 * k + 4 * t4);
        uint32_t xh[2][4], xm[2][4], xl[2][4];
#pragma unroll
        for (int e = 0; e < 2; ++e)
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                split_pair(win[e][h][o.x], win[e][h][o.y], xh[e][h], xm[e][h], xl[e][h]);
                split_pair(win[e][h][o.z], win[e][h][o.w], xh[e][2 + h], xm[e][2 + h], xl[e][2 + h]);
            }
#pragma unroll
        for (int j = 0; j < 6; j += 2) {
            uint32_t wh[2][2], wm[2][2], wl[2][2];
#pragma unroll
            for (int f = 0; f < 2; ++f) {
                const float4 v = *reinterpret_cast<const float4*>(wr + 8 * (j + f) * FWP + 16 * k);
                split_pair(v.x, v.y, wh[f][0], wm[f][0], wl[f][0]);
                split_pair(v.z, v.w, wh[f][1], wm[f][1], wl[f][1]);
            }
            mma_split(&acc[j], xh, xm, xl, wh, wm, wl);
        }
    }
    store(SPLIT_UNSCALE, false);
    if (__syncthreads_or(!finite)) {
#pragma unroll
        for (int e = 0; e < 2; ++e)
#pragma unroll
            for (int j = 0; j < 6; ++j)
#pragma unroll
                for (int i = 0; i < 4; ++i) acc[j][e][i] = 0.f;
#pragma unroll 1
        for (int k = 0; k < FK; ++k) {
            const int o = tbl[k];
#pragma unroll
            for (int j = 0; j < 6; ++j)
#pragma unroll
                for (int i = 0; i < 2; ++i) {
                    const float v = sw[(48 * nh + 8 * j + 2 * t4 + i) * FWP + k];
#pragma unroll
                    for (int e = 0; e < 2; ++e)
#pragma unroll
                        for (int h = 0; h < 2; ++h) acc[j][e][2 * h + i] = fmaf(win[e][h][o], v, acc[j][e][2 * h + i]);
                }
        }
        store(1.f, true);
        __syncthreads();
    }
    // the convolution's map (a tile's last row and column are also its neighbours' first)
    for (int i = tid; i < 2 * FPH * 2 * FPW * (FO / 4); i += 256) {
        const int px = i / (FO / 4), q = i - FO / 4 * px, r = px / (2 * FPW), c = px - 2 * FPW * r;
        const int oy = cy0 + r, ox = cx0 + c;
        if (oy >= p.OH || ox >= p.OW) continue;
        p.conv[(((size_t)img * p.OH + oy) * p.OW + ox) * (FO / 4) + q] = *reinterpret_cast<const float4*>(sy + (r * FCW + c) * FYP + 4 * q);
    }
    for (int i = tid; i < FPH * FPW * (FO / 4); i += 256) {
        const int px = i / (FO / 4), q = i - FO / 4 * px, r = px / FPW, c = px - FPW * r;
        const int py = FPH * ty + r, qx = FPW * tx + c;
        if (py >= p.PH || qx >= p.PW) continue;
        const float* src = sy + (2 * r * FCW + 2 * c) * FYP + 4 * q;
        float4 m = *reinterpret_cast<const float4*>(src);
#pragma unroll
        for (int a = 0; a < 3; ++a)
#pragma unroll
            for (int b = 0; b < 3; ++b) m = max4(m, *reinterpret_cast<const float4*>(src + (a * FCW + b) * FYP));
        if (!sqn_dbg_ok(2 * py + 2 < p.OH && 2 * qx + 2 < p.OW, p.status)) continue;
        p.pool[(((size_t)img * p.PH + py) * p.PW + qx) * (FO / 4) + q] = m;
    }
}

}  // namespace

// Stores the convolution's map at d.out and the pooled one at pool.  One CTA per SM at most: at 227 x 227 that is one image.
int launch_stem_small_f32(const ConvDesc& d, void* pool, cudaStream_t stream)
{
    StemF32Params p;
    std::memset(&p, 0, sizeof(p));
    if (d.K != 7 || d.S != 2 || d.pad != 0 || d.Cin != 3 || d.Cout != FO || !d.relu || d.out_c_total != FO || d.OH < 3 || d.OW < 3 ||
        (reinterpret_cast<uintptr_t>(d.bias) & 7u))
        return SQN_ERR_UNSUPPORTED;
    p.in = static_cast<const float*>(d.in); p.w = static_cast<const float*>(d.w); p.bias = d.bias;
    p.conv = static_cast<float4*>(d.out); p.pool = static_cast<float4*>(pool);
    p.status = device_status_word();
    p.H = d.H; p.W = d.W; p.OH = d.OH; p.OW = d.OW; p.PH = (d.OH - 3) / 2 + 1; p.PW = (d.OW - 3) / 2 + 1;
    const int tiles_y = (p.PH + FPH - 1) / FPH;
    p.tiles_x = (p.PW + FPW - 1) / FPW;
    p.tiles = tiles_y * p.tiles_x;
    // (the tiles of the pooled map have to cover the convolution's, and an image's offsets have to fit 32 bits)
    if (2 * FPH * tiles_y < p.OH || 2 * FPW * p.tiles_x < p.OW || (long long)p.H * p.W * 3 > 0x7fffffffLL || (long long)d.N * p.tiles > sm_count())
        return SQN_ERR_UNSUPPORTED;
    p.early = d.params_static;
    static SmemAttr attr;
    if (attr.allow((const void*)stem_small_f32_kernel, F_SMEM) != cudaSuccess) return SQN_ERR_CUDA;
    if (launch_chained(stem_small_f32_kernel, dim3((unsigned)(d.N * p.tiles)), dim3(256), F_SMEM, stream, p) != cudaSuccess) return SQN_ERR_CUDA;
    note_launch("stem_small_f32");
    return cudaGetLastError() == cudaSuccess ? SQN_OK : SQN_ERR_CUDA;
}

}  // namespace sqn
