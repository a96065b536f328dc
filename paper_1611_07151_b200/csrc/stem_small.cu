// The 16-bit stem (7x7/2 on 3 layers, 96 output layers) and the 3x3/2 max-pool behind it for few images, in one launch that
// stores both maps.
//
// At one image the stem is latency, not work.  Here a CTA takes 4 x 6 pooled pixels, i.e. 9 x 13 = 117 convolution pixels (140 CTAs for
// 227 x 227: one wave), as mma.sync tiles of 32 pixels x 48 layers per warp.  The input patch lies in shared memory as pixels of
// 8 bytes (three layers and the constant 1 that meets the bias folded into the kernels), so that the eight pixels of a kernel
// row are 64 consecutive bytes starting 16 bytes further per output column: ldmatrix reads the im2col rows where they lie.
// A caller's kernels are brought into that form by every CTA (in the time the grid ahead takes to finish).  One image per
// forward, back to back: 83 us with repack, convolution and pool as three launches, 74 with this one.
#include <cstring>

#include "f32_common.cuh"
#include "smem_attr.h"
#include "sqn_internal.h"
#include "tc_common.cuh"
#include "tc_host.h"

namespace sqn {
namespace {

constexpr int SO = 96;                          // output layers
constexpr int SPH = 4, SPW = 6;                 // pooled pixels of a CTA
constexpr int SCH = 2 * SPH + 1, SCW = 2 * SPW + 1;
constexpr int SPIX = SCH * SCW;                 // convolution pixels of a CTA (117 of 8 x 16)
constexpr int SXH = 2 * SCH + 5, SXW = 32;      // input rows, pixels per input row (2 * SCW + 5, and the zero kernel column)
constexpr int SXP = 272;                        // bytes per input row
constexpr int SWP = 464;                        // bytes per kernel row of 224 elements (an odd number of 16-byte units)
constexpr int SYP = 208;                        // bytes per convolution pixel (the same)
constexpr int S_OFF_X = SO * SWP, S_OFF_Y = S_OFF_X + SXH * SXP;
constexpr int S_SMEM = S_OFF_Y + 128 * SYP;
static_assert(SPIX <= 128 && 2 * SCW + 6 <= SXW, "");

struct StemSmallParams {
    const void* in;             // RAW: [N][H][W][3], else [N][Hp][Wp][4] with the constant 1
    const void* w;              // RAW: [96][7][7][3], else [96][7][8][4] with the bias
    const float* bias;          // (RAW)
    uint4* conv;                // [N][OH][OW][96]
    uint4* pool;                // [N][PH][PW][96]
    int* status;
    int H, W, Hp, Wp, OH, OW, PH, PW, tiles_x, tiles;       // tiles per image
    int early;                  // the kernels are not written by the grid ahead
};

template <bool F16>
__device__ __forceinline__ uint32_t max_x2(uint32_t a, uint32_t b)
{
    if (F16) {
        __half2 m = __hmax2(*reinterpret_cast<__half2*>(&a), *reinterpret_cast<__half2*>(&b));
        return *reinterpret_cast<uint32_t*>(&m);
    }
    __nv_bfloat162 m = __hmax2(*reinterpret_cast<__nv_bfloat162*>(&a), *reinterpret_cast<__nv_bfloat162*>(&b));
    return *reinterpret_cast<uint32_t*>(&m);
}

template <bool F16, bool RAW>
__global__ void __launch_bounds__(256) stem_small_kernel(const __grid_constant__ StemSmallParams p)
{
    extern __shared__ __align__(16) unsigned char sm_stem[];
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const uint32_t sm = (uint32_t)__cvta_generic_to_shared(sm_stem);
    const int img = (int)blockIdx.x / p.tiles, tile = (int)blockIdx.x - img * p.tiles;
    const int ty = tile / p.tiles_x, tx = tile - ty * p.tiles_x;
    const int cy0 = 2 * SPH * ty, cx0 = 2 * SPW * tx;           // first convolution pixel; the input patch starts at twice that
    chain_release();
    if (!p.early) chain_wait();
    if (RAW) {
        const unsigned short* w = static_cast<const unsigned short*>(p.w);
#pragma unroll 7
        for (int i = tid; i < SO * 56; i += 256) {              // kernel i / 56, pixel i % 56 of its 7 x 8
            const int m = i / 56, r = i - 56 * m, kh = r >> 3, px = r & 7;
            uint32_t lo = 0u, hi = 0u;
            if (px < 7) {
                const unsigned short* s = w + (m * 49 + kh * 7 + px) * 3;
                lo = (uint32_t)__ldg(s) | ((uint32_t)__ldg(s + 1) << 16);
                hi = (uint32_t)__ldg(s + 2);
            }
            if (r < 2) {
                const uint32_t hl = bias_hi_lo(__ldg(p.bias + m), F16);
                hi |= r == 0 ? hl << 16 : hl & 0xffff0000u;
            }
            *reinterpret_cast<uint2*>(sm_stem + m * SWP + 8 * r) = make_uint2(lo, hi);
        }
    } else {
        for (int i = tid; i < SO * 28; i += 256) {
            const int m = i / 28, r = i - 28 * m;
            cp_async_16(sm + (uint32_t)(m * SWP + 16 * r), static_cast<const unsigned short*>(p.w) + 224 * m + 8 * r, true);
        }
    }
    if (p.early) chain_wait();
    if (RAW) {
        const unsigned short* in = static_cast<const unsigned short*>(p.in) + (size_t)img * p.H * p.W * 3;
        const uint32_t one = F16 ? 0x3c000000u : 0x3f800000u;
#pragma unroll 3
        for (int i = tid; i < SXH * SXW; i += 256) {
            const int y = i / SXW, x = i - SXW * y, iy = 2 * cy0 + y, ix = 2 * cx0 + x;
            uint32_t lo = 0u, hi = 0u;
            if (iy < p.H && ix < p.W) {
                const unsigned short* s = in + (iy * p.W + ix) * 3;
                lo = (uint32_t)__ldg(s) | ((uint32_t)__ldg(s + 1) << 16);
                hi = (uint32_t)__ldg(s + 2) | one;
            }
            *reinterpret_cast<uint2*>(sm_stem + S_OFF_X + y * SXP + 8 * x) = make_uint2(lo, hi);
        }
    } else {
        const unsigned short* in = static_cast<const unsigned short*>(p.in) + (size_t)img * p.Hp * p.Wp * 4;
        for (int i = tid; i < SXH * SXW / 2; i += 256) {
            const int y = i / (SXW / 2), x = 2 * (i - SXW / 2 * y), iy = 2 * cy0 + y, ix = 2 * cx0 + x;
            const bool ok = iy < p.Hp && ix < p.Wp;             // (Wp is even: both pixels or neither)
            cp_async_16(sm + (uint32_t)(S_OFF_X + y * SXP + 8 * x), ok ? in + (iy * p.Wp + ix) * 4 : in, ok);
        }
        cp_async_commit();
        cp_async_wait<0>();
    }
    __syncthreads();

    // a warp: 32 pixels x 48 layers (the kernels are then read four times per CTA, not eight)
    const int mg = warp >> 1, nh = warp & 1;
    float acc[2][6][4];
#pragma unroll
    for (int e = 0; e < 2; ++e)
#pragma unroll
        for (int j = 0; j < 6; ++j)
#pragma unroll
            for (int i = 0; i < 4; ++i) acc[e][j][i] = 0.f;
    {
        uint32_t xa[2];
#pragma unroll
        for (int e = 0; e < 2; ++e) {
            int m = 32 * mg + 16 * e + (lane & 15);
            if (m >= SPIX) m = 0;                               // (rows past the tile: computed and dropped)
            const int r = m / SCW, c = m - SCW * r;
            xa[e] = sm + (uint32_t)(S_OFF_X + 2 * r * SXP + 16 * c + 16 * (lane >> 4));
        }
        const uint32_t wa = sm + (uint32_t)((48 * nh + ((lane >> 4) << 3) + (lane & 7)) * SWP + ((lane >> 3) & 1) * 16);
#pragma unroll 7
        for (int k = 0; k < 14; ++k) {                          // kernel row k / 2, half of its 32 elements
            uint32_t a[2][4];
#pragma unroll
            for (int e = 0; e < 2; ++e) ldmatrix_x4(a[e], xa[e] + (uint32_t)((k >> 1) * SXP + (k & 1) * 32));
#pragma unroll
            for (int j = 0; j < 3; ++j) {
                uint32_t b[4];
                ldmatrix_x4(b, wa + (uint32_t)(16 * j * SWP + 32 * k));
#pragma unroll
                for (int e = 0; e < 2; ++e) {
                    mma_16816<F16>(acc[e][2 * j], a[e], b[0], b[1]);
                    mma_16816<F16>(acc[e][2 * j + 1], a[e], b[2], b[3]);
                }
            }
        }
    }
    // ReLU and rounding, the convolution's pixels side by side
#pragma unroll
    for (int e = 0; e < 2; ++e) {
        unsigned char* y = sm_stem + S_OFF_Y + (32 * mg + 16 * e + (lane >> 2)) * SYP + 96 * nh + 4 * (lane & 3);
#pragma unroll
        for (int j = 0; j < 6; ++j) {
            *reinterpret_cast<uint32_t*>(y + 16 * j) = pack_relu_x2(acc[e][j][0], acc[e][j][1], F16);
            *reinterpret_cast<uint32_t*>(y + 8 * SYP + 16 * j) = pack_relu_x2(acc[e][j][2], acc[e][j][3], F16);
        }
    }
    __syncthreads();
    // the convolution's map (a tile's last row and column are also its neighbours' first)
    for (int i = tid; i < 2 * SPH * 2 * SPW * 12; i += 256) {
        const int px = i / 12, q = i - 12 * px, r = px / (2 * SPW), c = px - 2 * SPW * r;
        const int oy = cy0 + r, ox = cx0 + c;
        if (oy >= p.OH || ox >= p.OW) continue;
        p.conv[(((size_t)img * p.OH + oy) * p.OW + ox) * 12 + q] = *reinterpret_cast<const uint4*>(sm_stem + S_OFF_Y + (r * SCW + c) * SYP + 16 * q);
    }
    for (int i = tid; i < SPH * SPW * 12; i += 256) {
        const int px = i / 12, q = i - 12 * px, r = px / SPW, c = px - SPW * r;
        const int py = SPH * ty + r, qx = SPW * tx + c;
        if (py >= p.PH || qx >= p.PW) continue;
        const unsigned char* src = sm_stem + S_OFF_Y + (2 * r * SCW + 2 * c) * SYP + 16 * q;
        uint4 m = *reinterpret_cast<const uint4*>(src);
#pragma unroll
        for (int a = 0; a < 3; ++a)
#pragma unroll
            for (int b = 0; b < 3; ++b) {
                const uint4 v = *reinterpret_cast<const uint4*>(src + (a * SCW + b) * SYP);
                m.x = max_x2<F16>(m.x, v.x); m.y = max_x2<F16>(m.y, v.y); m.z = max_x2<F16>(m.z, v.z); m.w = max_x2<F16>(m.w, v.w);
            }
        if (!sqn_dbg_ok(2 * py + 2 < p.OH && 2 * qx + 2 < p.OW, p.status)) continue;
        p.pool[(((size_t)img * p.PH + py) * p.PW + qx) * 12 + q] = m;
    }
}

template <bool F16, bool RAW>
cudaError_t launch(const StemSmallParams& p, int blocks, cudaStream_t stream)
{
    static SmemAttr attr;
    const cudaError_t arc = attr.allow((const void*)stem_small_kernel<F16, RAW>, S_SMEM);
    if (arc != cudaSuccess) return arc;
    return launch_chained(stem_small_kernel<F16, RAW>, dim3((unsigned)blocks), dim3(256), (size_t)S_SMEM, stream, p);
}

}  // namespace

// d: the convolution; d.stem_prepacked: in and w have the packed layouts (params_static: w is not written by the launch ahead),
// else as the caller's.  Stores the convolution's map at d.out and the pooled one at pool.
int launch_stem_small(const ConvDesc& d, void* pool, cudaStream_t stream)
{
    StemSmallParams p;
    std::memset(&p, 0, sizeof(p));
    if (d.K != 7 || d.S != 2 || d.pad != 0 || d.Cin != 3 || d.Cout != SO || !d.relu || d.out_c_total != SO || d.OH < 3 || d.OW < 3)
        return SQN_ERR_UNSUPPORTED;
    p.in = d.in; p.w = d.w; p.bias = d.bias; p.conv = static_cast<uint4*>(d.out); p.pool = static_cast<uint4*>(pool);
    p.status = device_status_word();
    p.H = d.H; p.W = d.W; p.Hp = stem_packed_rows(d.H); p.Wp = stem_packed_cols(d.W);
    p.OH = d.OH; p.OW = d.OW; p.PH = (d.OH - 3) / 2 + 1; p.PW = (d.OW - 3) / 2 + 1;
    const int tiles_y = (p.PH + SPH - 1) / SPH;
    p.tiles_x = (p.PW + SPW - 1) / SPW;
    p.tiles = tiles_y * p.tiles_x;
    // One CTA per SM at most: at 227 x 227 that is one image.  Two images, with the repack as a launch of its own so that not every
    // CTA repeats it, were 1.6 us faster than the kernels below, three 2.4 us slower, eight 10.7 us.
    // (The tiles of the pooled map have to cover the convolution's, and a packed image's offsets have to fit 32 bits)
    if (2 * SPH * tiles_y < p.OH || 2 * SPW * p.tiles_x < p.OW || (long long)p.Hp * p.Wp * 4 > 0x7fffffffLL ||
        (long long)d.N * p.tiles > sm_count())
        return SQN_ERR_UNSUPPORTED;
    p.early = d.params_static;
    const int blocks = d.N * p.tiles;
    const cudaError_t rc = d.stem_prepacked ? (d.f16 ? launch<true, false>(p, blocks, stream) : launch<false, false>(p, blocks, stream))
                                            : (d.f16 ? launch<true, true>(p, blocks, stream) : launch<false, true>(p, blocks, stream));
    if (rc != cudaSuccess) return SQN_ERR_CUDA;
    note_launch("stem_small");
    return cudaGetLastError() == cudaSuccess ? SQN_OK : SQN_ERR_CUDA;
}

}  // namespace sqn
