// 16-bit convolution for small layers (one image, few pixels): implicit GEMM with the reduction split over the warps of a
// CTA, warp-level matrix instructions (mma.sync m16n8k16, fp32 accumulation).
//
// A layer of one image is a few microseconds of latency, not work: the tcgen05 kernels spend them on tensor maps, TMEM,
// barriers and hand-overs between roles (fire9 at one image, squeeze and both expands: 14.5 us there, 6.1 here; fire2 8.6,
// 6.1).  Here there is nothing to set up: every warp copies its own chunks of 32 reduction elements asynchronously into its
// own ring (16-byte pieces, rows of 80 bytes: no bank conflicts), waits for nobody else, multiplies the whole 32 x 32 output
// tile by them, and the warps' partial sums are added once at the end, in a fixed order, with bias and ReLU in fp32.  Two
// layers that read the same input (the expands of a fire layer) go out as one grid.
#include <cmath>
#include <cstring>

#include "f32_common.cuh"
#include "smem_attr.h"
#include "sqn_internal.h"
#include "tc_common.cuh"
#include "tc_host.h"

namespace sqn {
namespace {

constexpr int MK = 32;                  // reduction elements per chunk
constexpr int MT = 32;                  // output pixels and output layers per tile
constexpr int MPITCH = 80;              // bytes per operand row: 64 and 16 to keep rows of a fragment load in different banks
constexpr int MSLOT = 2 * MT * MPITCH;  // bytes of a ring slot: pixel rows, then kernel rows
constexpr int MRP = MT + 4;             // floats per row of partial sums

struct MmaSmallParams {
    const unsigned short* in;
    const unsigned short* w;
    const float* bias;
    unsigned short* out;
    int* status;
    int Cin, H, W, Cout, K, pad, OW, OHW, M, Kdim;
    int out_c_offset, out_c_total, relu;
    FastDiv div_ohw, div_ow, div_cin, div_k;
    int chunks;
    int n_tiles, blocks;
    int early;
};

template <bool F16, int SL, int ST>
__device__ __forceinline__ void conv_mma_small_body(const MmaSmallParams& p, const int bid)
{
    extern __shared__ __align__(16) unsigned char sm_mma[];
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int mt = bid / p.n_tiles, n0 = (bid - mt * p.n_tiles) * MT, m0 = mt * MT;
    const uint32_t sm = (uint32_t)__cvta_generic_to_shared(sm_mma);
    const uint32_t ring = sm + (uint32_t)(warp * ST * MSLOT);

    // this lane's copies: piece q (8 reduction elements) of rows r0 + 8 * j
    const int q = lane & 3, r0 = lane >> 2;
    int a_off[4], a_ih[4], a_iw[4];
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        const int m = m0 + r0 + 8 * j;
        if (m < p.M) {
            const int img = fast_div(m, p.div_ohw), r = m - img * p.OHW;
            const int oh = fast_div(r, p.div_ow), ow = r - oh * p.OW;
            a_ih[j] = oh - p.pad; a_iw[j] = ow - p.pad;
            a_off[j] = ((img * p.H + a_ih[j]) * p.W + a_iw[j]) * p.Cin;
        } else { a_off[j] = 0; a_ih[j] = -(1 << 30); a_iw[j] = 0; }
    }
    const uint32_t my_piece = (uint32_t)(r0 * MPITCH + 16 * q);
    auto load_w = [&](int ch, int slot) {
        const uint32_t dst = ring + (uint32_t)(slot * MSLOT + MT * MPITCH) + my_piece;
        const int k = ch * MK + 8 * q;
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const bool ok = k < p.Kdim && n0 + r0 + 8 * j < p.Cout;
            cp_async_16(dst + (uint32_t)(8 * j * MPITCH), ok ? p.w + (size_t)(n0 + r0 + 8 * j) * p.Kdim + k : p.w, ok);
        }
    };
    auto load_x = [&](int ch, int slot) {
        const uint32_t dst = ring + (uint32_t)(slot * MSLOT) + my_piece;
        const int k = ch * MK + 8 * q;
        const int t = fast_div(k, p.div_cin), c = k - t * p.Cin, kh = fast_div(t, p.div_k), kw = t - kh * p.K;
        const int off = (kh * p.W + kw) * p.Cin + c;
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const bool ok = k < p.Kdim && (unsigned)(a_ih[j] + kh) < (unsigned)p.H && (unsigned)(a_iw[j] + kw) < (unsigned)p.W;
            cp_async_16(dst + (uint32_t)(8 * j * MPITCH), ok ? p.in + (a_off[j] + off) : p.in, ok);
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
    float acc[2][4][4];
#pragma unroll
    for (int i = 0; i < 2; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j)
#pragma unroll
            for (int e = 0; e < 4; ++e) acc[i][j][e] = 0.f;
    // fragment addresses: pixels, rows (lane & 15) of a 16-row block, k half lane >> 4; kernels, rows of two 8-row blocks
    const uint32_t xf = ring + (uint32_t)((lane & 15) * MPITCH + (lane >> 4) * 16);
    const uint32_t wf = ring + (uint32_t)(MT * MPITCH + (((lane >> 4) << 3) + (lane & 7)) * MPITCH + ((lane >> 3) & 1) * 16);
    for (int i = 0, slot = 0; i < mine; ++i) {
        cp_async_wait<ST - 2>();
        __syncwarp();                   // chunk i is here for every lane, and every lane has done with chunk i - 1's slot
        {
            const int nx = i + ST - 1, ns = slot == 0 ? ST - 1 : slot - 1;
            if (nx < mine) { load_w(warp + SL * nx, ns); load_x(warp + SL * nx, ns); }
            cp_async_commit();
        }
#pragma unroll
        for (int k = 0; k < 2; ++k) {
            uint32_t a[2][4], b[2][4];
#pragma unroll
            for (int e = 0; e < 2; ++e) {
                ldmatrix_x4(a[e], xf + (uint32_t)(slot * MSLOT + e * 16 * MPITCH + k * 32));
                ldmatrix_x4(b[e], wf + (uint32_t)(slot * MSLOT + e * 16 * MPITCH + k * 32));
            }
#pragma unroll
            for (int e = 0; e < 2; ++e)
#pragma unroll
                for (int f = 0; f < 4; ++f) mma_16816<F16>(acc[e][f], a[e], b[f >> 1][2 * (f & 1)], b[f >> 1][2 * (f & 1) + 1]);
        }
        if (++slot == ST) slot = 0;
    }
    cp_async_wait<0>();
    __syncwarp();
    // partial sums into the warp's own ring, then all warps' sums in order: eight layers of a pixel per thread
    static_assert(MT * MRP * 4 <= ST * MSLOT, "the partial sums fit the ring");
    float* part = reinterpret_cast<float*>(sm_mma + warp * ST * MSLOT);
#pragma unroll
    for (int e = 0; e < 2; ++e)
#pragma unroll
        for (int f = 0; f < 4; ++f) {
            float* d = part + (16 * e + (lane >> 2)) * MRP + 8 * f + 2 * (lane & 3);
            *reinterpret_cast<float2*>(d) = make_float2(acc[e][f][0], acc[e][f][1]);
            *reinterpret_cast<float2*>(d + 8 * MRP) = make_float2(acc[e][f][2], acc[e][f][3]);
        }
    __syncthreads();
    for (int i = tid; i < MT * MT / 8; i += 32 * SL) {
        const int r = i >> 2, l8 = 8 * (i & 3);
        const int m = m0 + r, n = n0 + l8;
        if (m >= p.M || n >= p.Cout) continue;
        float4 v0 = make_float4(0.f, 0.f, 0.f, 0.f), v1 = v0;
#pragma unroll
        for (int s = 0; s < SL; ++s) {
            const float4* src = reinterpret_cast<const float4*>(sm_mma + s * ST * MSLOT + (r * MRP + l8) * 4);
            const float4 q0 = src[0], q1 = src[1];
            v0.x += q0.x; v0.y += q0.y; v0.z += q0.z; v0.w += q0.w;
            v1.x += q1.x; v1.y += q1.y; v1.z += q1.z; v1.w += q1.w;
        }
        const float4 b0 = __ldg(reinterpret_cast<const float4*>(p.bias + n)), b1 = __ldg(reinterpret_cast<const float4*>(p.bias + n) + 1);
        v0.x += b0.x; v0.y += b0.y; v0.z += b0.z; v0.w += b0.w;
        v1.x += b1.x; v1.y += b1.y; v1.z += b1.z; v1.w += b1.w;
        if (!sqn_dbg_ok(m >= 0 && p.out_c_offset + n + 8 <= p.out_c_total, p.status)) continue;
        uint4 o;
        if (p.relu) o = make_uint4(pack_relu_x2(v0.x, v0.y, F16), pack_relu_x2(v0.z, v0.w, F16), pack_relu_x2(v1.x, v1.y, F16), pack_relu_x2(v1.z, v1.w, F16));
        else o = make_uint4(pack_x2(v0.x, v0.y, F16), pack_x2(v0.z, v0.w, F16), pack_x2(v1.x, v1.y, F16), pack_x2(v1.z, v1.w, F16));
        *reinterpret_cast<uint4*>(p.out + (size_t)m * p.out_c_total + p.out_c_offset + n) = o;
    }
}

template <bool F16, int SL, int ST>
__global__ void __launch_bounds__(32 * SL)
conv_mma_small_kernel(const __grid_constant__ MmaSmallParams p0, const __grid_constant__ MmaSmallParams p1)
{
    chain_release();
    if ((int)blockIdx.x < p0.blocks) conv_mma_small_body<F16, SL, ST>(p0, (int)blockIdx.x);
    else conv_mma_small_body<F16, SL, ST>(p1, (int)blockIdx.x - p0.blocks);
}

bool fill(const ConvDesc& d, MmaSmallParams* p)
{
    std::memset(p, 0, sizeof(*p));
    const long long M = (long long)d.N * d.OH * d.OW, Kdim = (long long)d.K * d.K * d.Cin;
    if (M > 0x3fffffffLL || (long long)d.N * d.H * d.W * d.Cin > 0x3fffffffLL || d.pad > 1024 || (long long)d.W * d.Cin > 0xfffff) return false;
    p->in = static_cast<const unsigned short*>(d.in); p->w = static_cast<const unsigned short*>(d.w); p->bias = d.bias;
    p->out = static_cast<unsigned short*>(d.out); p->status = device_status_word();
    p->Cin = d.Cin; p->H = d.H; p->W = d.W; p->Cout = d.Cout; p->K = d.K; p->pad = d.pad;
    p->OW = d.OW; p->OHW = d.OH * d.OW; p->M = (int)M; p->Kdim = (int)Kdim;
    p->out_c_offset = d.out_c_offset; p->out_c_total = d.out_c_total; p->relu = d.relu;
    p->div_ohw = make_div(p->OHW); p->div_ow = make_div(p->OW); p->div_cin = make_div(p->Cin); p->div_k = make_div(p->K);
    p->chunks = (p->Kdim + MK - 1) / MK;
    p->n_tiles = (d.Cout + MT - 1) / MT;
    const long long blocks = ((M + MT - 1) / MT) * p->n_tiles;
    if (blocks > 0x3fffffffLL) return false;
    p->blocks = (int)blocks;
    p->early = d.params_static;
    return true;
}

template <bool F16, int SL, int ST>
cudaError_t launch(const MmaSmallParams& a, const MmaSmallParams& b, cudaStream_t stream)
{
    constexpr size_t smem = (size_t)SL * ST * MSLOT;
    static SmemAttr attr;
    const cudaError_t arc = attr.allow((const void*)conv_mma_small_kernel<F16, SL, ST>, smem);
    if (arc != cudaSuccess) return arc;
    const cudaError_t rc =
        launch_chained(conv_mma_small_kernel<F16, SL, ST>, dim3((unsigned)(a.blocks + b.blocks)), dim3(32 * SL), smem, stream, a, b);
    if (rc == cudaSuccess) note_launch("conv_mma_small%s, %d warps, %d slots", b.blocks ? " x 2" : "", SL, ST);
    return rc;
}

// Warps that share a tile's reduction and ring slots per warp: no more warps than chunks, and as many slots as let all CTAs
// of the launch be resident (122 KB a CTA up to one per SM, 82 KB up to two, 61 KB up to three, else 41 KB).  Deeper rings
// were no faster (fire9's 3x3 expand at one image: 3.3 us with two, three and five slots), fewer warps slower (4 warps 4.0 us).
template <bool F16>
cudaError_t launch_shape(const MmaSmallParams& a, const MmaSmallParams& b, cudaStream_t stream)
{
    const int chunks = b.blocks && b.chunks > a.chunks ? b.chunks : a.chunks, blocks = a.blocks + b.blocks, sms = sm_count();
    if (chunks == 1) return launch<F16, 1, 2>(a, b, stream);
    if (chunks == 2) return launch<F16, 2, 2>(a, b, stream);
    if (chunks <= 4 || blocks > 3 * sms) return launch<F16, 4, 2>(a, b, stream);
    if (blocks > 2 * sms) return launch<F16, 4, 3>(a, b, stream);
    if (blocks > sms) return launch<F16, 8, 2>(a, b, stream);
    return launch<F16, 8, 3>(a, b, stream);
}

}  // namespace

// Time of the n layers as one launch, in microseconds.  Fitted to the layers of SqueezeNet and of a residual bottleneck at 1 to
// 8 images (within 15 %): a launch and its latencies, the chain of chunks in a warp, the tiles' set-up and stores, their MMAs.
float mma_small_estimate(const ConvDesc* d, int n)
{
    float tiles = 0.f, work = 0.f, kdim = 0.f;
    for (int i = 0; i < n; ++i) {
        if (d[i].S != 1 || d[i].pool || (reinterpret_cast<uintptr_t>(d[i].bias) & 15u)) return 1e30f;
        const float k = (float)d[i].K * d[i].K * d[i].Cin;
        const float t = ceilf((float)d[i].N * d[i].OH * d[i].OW / MT) * ((d[i].Cout + MT - 1) / MT);
        tiles += t;
        work += t * ceilf(k / MK);
        kdim = fmaxf(kdim, k);
    }
    return 1.9f + 0.0021f * kdim + 0.004f * tiles + 0.00025f * work;
}

int launch_conv_mma_small(const ConvDesc* d, int n, cudaStream_t stream)
{
    MmaSmallParams p[2];
    for (int i = 0; i < n; ++i)
        if ((reinterpret_cast<uintptr_t>(d[i].bias) & 15u) || !fill(d[i], &p[i])) return SQN_ERR_UNSUPPORTED;
    if (n == 1) { p[1] = p[0]; p[1].blocks = 0; }
    const cudaError_t rc = d[0].f16 ? launch_shape<true>(p[0], p[1], stream) : launch_shape<false>(p[0], p[1], stream);
    if (rc != cudaSuccess) return SQN_ERR_CUDA;
    return cudaGetLastError() == cudaSuccess ? SQN_OK : SQN_ERR_CUDA;
}

}  // namespace sqn
