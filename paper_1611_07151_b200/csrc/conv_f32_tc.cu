// fp32 convolution layer on the tensor cores, at fp32 precision: implicit GEMM, every fp32 operand written as the sum of
// three bf16 numbers, which is exact (3 x 8 significand bits).
//
//   x = x0 + x1 + x2,  w = w0 + w1 + w2:   w*x = w0*x0 + (w0*x1 + w1*x0) + (w0*x2 + w1*x1 + w2*x0) + dropped
//
// x0 is x rounded to nearest (the remainder is below 2^-8 of x and of either sign), x1 the leading eight bits of the
// remainder, x2 the rest; the dropped products w1*x2, w2*x1, w2*x2 are of either sign, 0.23 units of 2^-24 of w*x in the root mean
// square and up to 1.75 (four million random pairs; the rounding of one fp32 multiply-add: 0.42, up to 1), so that an output that
// is a single product may be off by more than a multiply-add's, a sum is not.  The products are exact in the tensor core; its
// accumulator, though, cuts sums off at 24 bits instead of rounding them: an error towards zero that would grow with the
// length of the reduction and add up from layer to layer.  So w0*x0 is summed on the tensor core over short segments of
// the reduction only (32 elements; 64 would take 10 % less time), which the epilogue warps add up in registers with rounded
// fp32 additions, and what a segment loses on average is added back (FT_CUT); the other five products are 2^-8 smaller and
// stay in an accumulator of their own for the whole tile.  Relative 2-norm error of a layer against 64-bit arithmetic: 0.7e-7
// to 2e-7 (multiply-adds in sequence: 2e-7 to 1e-6); of SqueezeNet's logits at batch 160: 1.05e-7 (1.13e-7).
// Operands are scaled by 2^16 before the split (SPLIT_SCALE; SqueezeNet in fp32, 256 images: 5458 us without it, 5478 with), so that it is exact for every number below 2^112.
// Outputs that are not finite, or too large for the scaled sums, are computed again with fp32 multiply-adds.
//
// GEMM view: D[layer][pixel] = sum_k W[layer][k] * X[pixel][k].  The kernels are the M = 128 operand and sit in TMEM, the
// N = 128 pixels of a tile are the shared-memory operand: with both in shared memory a 128 x 128 x 16 MMA alone takes the
// shared memory's whole bandwidth (8 KB in 64 clocks), and the split below needs some of it.  Any K, stride, padding and
// layer counts.  Where the pixel operand of a tile comes from:
//   FLAT    1x1, stride 1, no padding, Cin a multiple of 4: TMA boxes of 128 pixels x 32 layers
//   PATCH   K > 1, stride 1, Cin a multiple of 4: the tile is 128 consecutive positions of the maps laid out with `pad` zero
//           columns after every row and `pad` zero rows after every map (the padding of both neighbours), so that tap
//           (kh, kw) reads the same positions shifted by a constant: every pixel is loaded and split once per tile, not
//           once per tap, and a tap is an MMA whose descriptor starts that many rows further into the split patch
//   BOX     anything else: the input window of a tile of bw x bh output pixels is staged in shared memory as it is (zeros
//           outside the map), im2col rows are read from there through a table of offsets
// What bounds it (clock traces and ablations at batch 256): instructions.  28 warps in six roles run straight-line code that
// does not stay in the schedulers' instruction caches, some six clocks per instruction and warp, so a unit costs what the
// slowest role's instructions for it cost: the issuing warp 1300 clocks (its 12 MMAs: 830), the splitting groups 1000 to 1350,
// the epilogue 1000; and once per tile 3200 to 4200 for bias, ReLU and stores, during which the two segment accumulators
// cover two units.  Against the FFMA kernel, batch 256: conv1 1053 us (2687), fire2's expand-3x3 234 (373), fire4's 359
// (1296), fire6's 299 (675), fire8's 316 (1237), conv10 290 (1256), fire8's squeeze 112 (234), fire4's expand-1x1 89 (204).
// Warps (one persistent CTA per SM, all of its tiles in one column of output layers):
//   0..7    two groups of four split pixels into bf16 planes, written as swizzled K-major operand tiles (FLAT, BOX: the
//           groups take the chunks of 32 reduction elements in turn; PATCH: each takes half of the patch's rows)
//   8..15   two groups of four split kernels into TMEM, the units (32 reduction elements of a tap) in turn: an output layer
//           per thread; once per CTA where the reduction is short, else streamed
//   16..23  epilogue: an output layer per thread, half of the tile's pixels per group of four; segment sums TMEM ->
//           registers, then bias, ReLU and stores of 32 consecutive layers of a pixel per warp
//   24, 25  TMA producers: pixels, kernels                 (26 idle: registers go by warpgroup)
//   27      MMA issuer (one elected lane), on the scheduler with the least other work
#include <cstring>

#include "f32_common.cuh"
#include "ptx_sm100.cuh"
#include "smem_attr.h"
#include "sqn_internal.h"
#include "tc_common.cuh"
#include "tc_host.h"

namespace sqn {
namespace {

using namespace ptx;

constexpr int FT_GT = 128;                  // threads of a group
constexpr int FT_W_KER = 8, FT_W_EPI = 16, FT_W_TMAX = 24, FT_W_TMAW = 25, FT_W_MMA = 27;       // first warps of the roles
constexpr int FT_THREADS = 32 * 28;
constexpr int FT_N = 128;                   // pixels (positions) per tile
constexpr int FT_BK = 32;                   // reduction elements per chunk, rows of 64 bytes in a bf16 plane
constexpr int FT_ROW = FT_BK * 2;
constexpr int FT_NA = FT_N * FT_BK / 4 / FT_GT;     // 16-byte pieces of 128 rows per thread of a group: 8
constexpr int FT_MAX_RA = 4, FT_MAX_SA = 4, FT_MAX_SB = 3;
// What the accumulator cuts off a segment on average, relative to it (measured over a layer: 1e-8 to 2.5e-8 on kernels of
// both signs, up to 4e-8 on sums of one sign); added back with the corrections.  Less than half a unit in the last place of
// any sum, so a sum that was exact stays as it is.
constexpr float FT_CUT = 1.6e-8f;
constexpr int FT_KSLOTS = 2;                // kernel slots in TMEM, one per kernel group
constexpr unsigned FT_COL_GX = 256, FT_COL_W = 384, FT_W_COLS = 48;     // TMEM: two segment accumulators, corrections, kernel slots
constexpr int FT_TBL_MAX = 2048;            // BOX: reduction elements per block of layers
constexpr size_t FT_SMEM_LIMIT = 227 * 1024;

enum { FT_FLAT = 0, FT_PATCH = 1, FT_BOX = 2 };
// Kernels: split once per CTA and kept packed in shared memory; streamed for every tile by TMA boxes; streamed by copies of
// 4 bytes (BOX, where the rows are no TMA tensor).
enum { FT_W_PACKED = 0, FT_W_BOXES = 1, FT_W_COPIES = 2 };

struct F32TcParams {
    const float* in;
    const float* w;
    const float* bias;
    float* out;
    int* status;
    int N, Cin, H, W, Cout, K, S, pad, OH, OW, OHW;
    int M, Kdim;                // output pixels, length of the reduction
    int out_c_offset, out_c_total, relu;
    FastDiv div_ohw, div_ow;    // output pixel -> (image, row, column)
    FastDiv div_pos, div_p;     // PATCH: position -> (image, padded row, padded column)
    int P, HP;                  // PATCH: positions per row, rows per map
    int mode;
    int n_tiles, n_step;        // columns of tiles, output layers per column (at most 128)
    int m_tiles, m_step;        // CTA b takes column b % n_tiles, pixel tiles b / n_tiles + i * m_step
    int grid;
    int taps;                   // taps that share a pixel chunk: K*K (PATCH) or 1
    int chunks, ksteps_last;    // pixel chunks of a tile, MMA k-steps of the last one
    int seg;                    // (chunk, tap) units whose w0*x0 products are summed on the tensor core before they are added in registers
    int kres;                   // 1: at most FT_KSLOTS units: the kernels stay in TMEM
    int tstore;                 // FLAT and BOX where vec_store holds and Cout is a multiple of 4: pixels per TMA store of the epilogue, 16, 32 or 64 (0: no TMA)
    int vec_store;              // 1: output rows and this layer's slice are 16-byte aligned
    int early;                  // 1: kernels and bias may be read before the wait for the grid ahead
    int ra, sa, sb;             // slots: split pixels, pixel boxes, kernel boxes
    int wsrc;                   // where a unit's split kernels come from, see FT_W_*
    int wrows;                  // FT_W_PACKED: rows (output layers) kept, a multiple of 32
    int khalf;                  // 1: every unit has 16 reduction elements only
    int prow;                   // rows of a pixel slot: 128, or those of a patch
    // BOX
    int bw_shift, bh;           // tile of (1 << bw_shift) x bh output pixels
    int tiles_w, tiles_h;
    int rh, rc, pitch;          // rows, pixels per row, floats per row of a box
    int stepb;                  // box pixels between windows: min(S, K) (pixels between windows are left out)
    int cb, nb, cpb;            // layers per block, blocks, chunks per block
    int box_vec;                // 1: 16-byte pieces
    FastDiv div_cb, div_tw, div_th, div_wrows, div_taps;
    unsigned plane_a, slot_a;   // bytes of a plane of a pixel slot, of a pixel slot
    unsigned stage_a;           // bytes of a pixel box (PATCH: of all rows of a patch)
    unsigned off_sa, off_sb, off_epi, off_tbl, off_ctl;
};

struct F32TcShared {
    unsigned long long a_full[FT_MAX_RA], a_empty[FT_MAX_RA];
    unsigned long long sa_full[FT_MAX_SA], sa_empty[FT_MAX_SA];
    unsigned long long sb_full[FT_MAX_SB], sb_empty[FT_MAX_SB];
    unsigned long long k_full[FT_KSLOTS];
    // done[u % 4]: the MMAs of unit u of the CTA's sequence have finished.  One commit per unit serves the kernel groups (slot
    // u % 2 is free), the pixel groups of FLAT and BOX (a chunk is a unit) and the epilogue (a segment ends with a unit): each
    // waits for units in order and none can be passed by four units, so two phases are never confused.
    unsigned long long done[4];
    unsigned long long seg_empty[2];
    unsigned long long gx_empty;
    unsigned tmem_base;
    volatile int abort_flag;
};

// The same question as mbar_try_wait's, answered at once
__device__ __forceinline__ bool mbar_test_wait(uint32_t bar, uint32_t parity)
{
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.test_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(ok)
        : "r"(bar), "r"(parity)
        : "memory");
    return ok != 0;
}
__device__ __forceinline__ void bar_sync(int id, int threads) { asm volatile("bar.sync %0, %1;" ::"r"(id), "r"(threads) : "memory"); }

// Four consecutive reduction elements -> the three planes (plane pitch in bytes), at address a of the first
__device__ __forceinline__ void store_split(uint32_t a, uint32_t pitch, float4 v)
{
    uint32_t h0, m0, l0, h1, m1, l1;
    split_pair(v.x, v.y, h0, m0, l0);
    split_pair(v.z, v.w, h1, m1, l1);
    asm volatile("st.shared.v2.b32 [%0], {%1, %2};" ::"r"(a), "r"(h0), "r"(h1) : "memory");
    asm volatile("st.shared.v2.b32 [%0], {%1, %2};" ::"r"(a + pitch), "r"(m0), "r"(m1) : "memory");
    asm volatile("st.shared.v2.b32 [%0], {%1, %2};" ::"r"(a + 2u * pitch), "r"(l0), "r"(l1) : "memory");
}
// Offset of quad q (four reduction elements, 8 bytes) of row r in a plane: rows of 64 bytes in the 64-byte swizzle
__device__ __forceinline__ uint32_t quad_offset(int r, int q)
{
    return (uint32_t)r * FT_ROW + ((((uint32_t)q >> 1) ^ (((uint32_t)r >> 1) & 3u)) << 4) + (((uint32_t)q & 1u) << 3);
}

__device__ __forceinline__ float4 ld_shared_v4(uint32_t a)
{
    float4 v;
    asm volatile("ld.shared.v4.f32 {%0, %1, %2, %3}, [%4];" : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w) : "r"(a) : "memory");
    return v;
}
__device__ __forceinline__ void ld_shared_u4(uint32_t a, uint32_t* v)
{
    asm volatile("ld.shared.v4.b32 {%0, %1, %2, %3}, [%4];" : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]) : "r"(a) : "memory");
}
__device__ __forceinline__ float ld_shared_f32(uint32_t a)
{
    float v;
    asm volatile("ld.shared.f32 %0, [%1];" : "=f"(v) : "r"(a) : "memory");
    return v;
}

// 16 consecutive 32-bit columns of this warp's 32 lanes, from registers
__device__ __forceinline__ void tmem_st_x16(uint32_t taddr, const uint32_t (&v)[16])
{
    asm volatile(
        "tcgen05.st.sync.aligned.32x32b.x16.b32 [%0], "
        "{%1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, %16};"
        ::"r"(taddr), "r"(v[0]), "r"(v[1]), "r"(v[2]), "r"(v[3]), "r"(v[4]), "r"(v[5]), "r"(v[6]), "r"(v[7]), "r"(v[8]), "r"(v[9]),
          "r"(v[10]), "r"(v[11]), "r"(v[12]), "r"(v[13]), "r"(v[14]), "r"(v[15])
        : "memory");
}
__device__ __forceinline__ void tmem_st_x8(uint32_t taddr, const uint32_t (&v)[16])        // (the first eight)
{
    asm volatile("tcgen05.st.sync.aligned.32x32b.x8.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};"
                 ::"r"(taddr), "r"(v[0]), "r"(v[1]), "r"(v[2]), "r"(v[3]), "r"(v[4]), "r"(v[5]), "r"(v[6]), "r"(v[7])
                 : "memory");
}
__device__ __forceinline__ void tmem_st_wait() { asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory"); }

// D[tmem] (+)= A[tmem] * B[smem]; bf16 operands, fp32 accumulate; issued by one thread.
__device__ __forceinline__ void mma_bf16_ts(uint32_t d_tmem, uint32_t a_tmem, uint64_t b_desc, uint32_t idesc, uint32_t accumulate)
{
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "setp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::1.kind::f16 [%0], [%1], %2, %3, p;\n\t}"
        ::"r"(d_tmem), "r"(a_tmem), "l"(b_desc), "r"(idesc), "r"(accumulate)
        : "memory");
}

// a + (a * c + b) for two fp32 numbers at a time, each operation rounded to nearest (half the instructions of the segments'
// sums: batch 256, fire8's expand-3x3 342 -> 314 us, conv10 316 -> 284)
__device__ __forceinline__ void add_cut2(float& ax, float& ay, uint64_t c, uint32_t bx, uint32_t by)
{
    asm("{\n\t.reg .b64 a, b, t;\n\t"
        "mov.b64 a, {%0, %1};\n\t"
        "mov.b64 b, {%3, %4};\n\t"
        "fma.rn.f32x2 t, a, %2, b;\n\t"
        "add.rn.f32x2 a, a, t;\n\t"
        "mov.b64 {%0, %1}, a;\n\t}"
        : "+f"(ax), "+f"(ay) : "l"(c), "r"(bx), "r"(by));
}

// Called by an epilogue warp, lane l with output layer n = (the first one's) + l (also past the last one).  m < 0: the sum of the
// absolute values of the layer's kernel.  Else output pixel m: as it is stored where the sums of the absolute values of its operands
// (ws: the kernel's) bound every partial sum, else with fp32 multiply-adds.  All lanes work on one pixel, four layers at a time, so
// that kernels are read in whole lines.  64 images of 128 -> 128 3x3 at 27 x 27 (90 us): with one infinity in all 513 us, in each image
// 780, while every output of such a warp was computed again 10030 and 14380 us (the FFMA kernel: 384).  A mask of the outputs made in the
// epilogue, a call with more in it, or this done behind the epilogue's loop or by other warps makes that loop spill: the stem of 256
// images 8 to 11 % slower.
__device__ __noinline__ float redo_output(const F32TcParams& p, int m, int n, float ws)
{
    const int lane = threadIdx.x & 31, first = n - lane;
    const int end = (first / p.n_step + 1) * p.n_step, left = (end < p.Cout ? end : p.Cout) - first;
    auto warp_sum = [](float v) {
#pragma unroll
        for (int h = 16; h > 0; h >>= 1) v += __shfl_xor_sync(0xffffffffu, v, h);
        return v;
    };
    const int row_len = p.K * p.Cin, map_row = p.W * p.Cin;
    float mine = 0.f;
    unsigned mask = left < 32 ? (1u << left) - 1u : 0xffffffffu;
    const float* x = p.in;
    int ih0 = 0, col0 = 0;                              // first row of the window, its first column in elements
    if (m >= 0) {
        const int img = fast_div(m, p.div_ohw), r = m - img * p.OHW, oh = fast_div(r, p.div_ow);
        const int iw0 = (r - oh * p.OW) * p.S - p.pad;
        ih0 = oh * p.S - p.pad;
        col0 = (iw0 < -p.K ? -p.K : iw0 < p.W ? iw0 : p.W) * p.Cin;        // (outside the map all the same: padding may be any number)
        x += (size_t)img * p.H * map_row;
        float xs = 0.f;
        for (int kh = 0; kh < p.K; ++kh) {
            if ((unsigned)(ih0 + kh) >= (unsigned)p.H) continue;
            const float* row = x + (size_t)(ih0 + kh) * map_row;
#pragma unroll 4
            for (int f = lane; f < row_len; f += 32) xs += (unsigned)col0 + (unsigned)f < (unsigned)map_row ? fabsf(__ldg(row + col0 + f)) : 0.f;
        }
        __syncwarp();
        xs = warp_sum(xs);
        if (lane < left) mine = __ldcg(p.out + (size_t)m * p.out_c_total + p.out_c_offset + n);      // (not through the L1: TMA may have stored it)
        mask &= __ballot_sync(0xffffffffu, !(xs < 0x1p111f && ws < 0x1p111f && xs * ws < 0x1p95f));
    }
    while (mask) {
        int l[4];
        float s[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            l[i] = mask ? __ffs(mask) - 1 : l[0];
            mask &= mask - 1u;
            s[i] = 0.f;
        }
        const float* w = p.w + (size_t)first * p.Kdim;
        for (int kh = 0; kh < p.K; ++kh, w += row_len) {
            const bool in = m >= 0 && (unsigned)(ih0 + kh) < (unsigned)p.H;
            const float* row = x + (size_t)(in ? ih0 + kh : 0) * map_row + col0;
#pragma unroll 2
            for (int f = lane; f < row_len; f += 32) {
                const float q = in && (unsigned)col0 + (unsigned)f < (unsigned)map_row ? __ldg(row + f) : 0.f;
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    const float v = __ldg(w + (size_t)l[i] * p.Kdim + f);
                    s[i] = m < 0 ? s[i] + fabsf(v) : fmaf(q, v, s[i]);
                }
            }
        }
        __syncwarp();
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const float v = warp_sum(s[i]);
            if (lane != l[i]) continue;
            mine = v;
            if (m >= 0) mine += __ldg(p.bias + n);
            if (m >= 0 && p.relu) mine = fmaxf(mine, 0.f);
        }
    }
    return mine;
}

// MODE is a compile-time constant so that a kernel's code stays small: six roles run different code at the same time, and
// with all modes and twice as much unrolled epilogue in one kernel they evicted one another from the instruction cache
// (expand-3x3 of fire2 at batch 256: 413 us instead of 300 at the time).
template <int MODE>
__device__ __forceinline__ void conv_f32_tc_body(const CUtensorMap& tmX, const CUtensorMap& tmW, const CUtensorMap& tmO, const F32TcParams& p, const int bid)
{
    extern __shared__ unsigned char smem_raw[];
    const uint32_t raw = smem_u32(smem_raw);
    const uint32_t base = (raw + 1023u) & ~1023u;
    unsigned char* base_ptr = smem_raw + (base - raw);
    F32TcShared* sh = reinterpret_cast<F32TcShared*>(base_ptr + p.off_ctl);
    int2* tbl = reinterpret_cast<int2*>(base_ptr + p.off_tbl);      // BOX: reduction element of a block -> {box offset, kernel offset or -1}

    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int nt = bid % p.n_tiles, mt0 = bid / p.n_tiles;
    const int n0 = nt * p.n_step;
    const int n_live = p.Cout - n0 < p.n_step ? p.Cout - n0 : p.n_step;     // output layers of this CTA
    const int my_tiles = mt0 < p.m_tiles ? (p.m_tiles - mt0 + p.m_step - 1) / p.m_step : 0;
    const int live_quads = (n_live + 31) >> 5;

    if (tid == 0) {
        const int px_warps = MODE == FT_PATCH ? 8 : 4;
        for (int s = 0; s < FT_MAX_RA; ++s) { mbar_init(smem_u32(&sh->a_full[s]), px_warps); mbar_init(smem_u32(&sh->a_empty[s]), 1); }
        for (int s = 0; s < FT_MAX_SA; ++s) { mbar_init(smem_u32(&sh->sa_full[s]), 1); mbar_init(smem_u32(&sh->sa_empty[s]), px_warps); }
        for (int s = 0; s < FT_MAX_SB; ++s) { mbar_init(smem_u32(&sh->sb_full[s]), 1); mbar_init(smem_u32(&sh->sb_empty[s]), 4); }
        for (int s = 0; s < FT_KSLOTS; ++s) { mbar_init(smem_u32(&sh->k_full[s]), 4); }
        for (int u = 0; u < 4; ++u) mbar_init(smem_u32(&sh->done[u]), 1);
        for (int a = 0; a < 2; ++a) mbar_init(smem_u32(&sh->seg_empty[a]), 2 * live_quads);
        mbar_init(smem_u32(&sh->gx_empty), 2 * live_quads);
        sh->abort_flag = 0;
        fence_mbar_init();
        if (p.sa) prefetch_tensormap(&tmX);
        if (p.wsrc == FT_W_BOXES) prefetch_tensormap(&tmW);
        if (MODE != FT_PATCH && p.tstore) prefetch_tensormap(&tmO);
    }
    if (warp == FT_W_MMA) {
        tmem_alloc(smem_u32(&sh->tmem_base), 512);
        tmem_relinquish();
        chain_release();            // (only once this CTA holds its TMEM: see conv_tc_body)
    }
    if (MODE == FT_BOX)
        for (int k = tid; k < p.cpb * FT_BK; k += FT_THREADS) {
            const int t = k / p.cb, c = k - t * p.cb, kh = t / p.K, kw = t - kh * p.K;
            tbl[k] = kh < p.K ? make_int2(kh * p.pitch + kw * p.cb + c, t * p.Cin + c) : make_int2(0, -1);
        }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem_base = sh->tmem_base;
    volatile int* abort_flag = &sh->abort_flag;
    const uint32_t done = smem_u32(sh->done);
    auto wait_done = [&](int u) {           // all lanes of a warp; units before the first have finished
        return u < 0 || __all_sync(0xffffffffu, wait_bar(done + 8u * ((uint32_t)u & 3u), ((uint32_t)u >> 2) & 1u, abort_flag, p.status));
    };
    // Global memory that the grid ahead may have written or may still read is touched after chain_wait() only.

    if (warp < FT_W_KER) {
        // ------------------------------------------------------------------ pixels
        asm volatile("setmaxnreg.dec.sync.aligned.u32 64;");
        const int grp = warp >> 2, gt = tid & (FT_GT - 1);
        const int q = gt & 7, r0 = gt >> 3;             // thread -> quad q of a chunk, rows r0 + 16 * j
        const uint32_t my_quad = quad_offset(r0, q);    // (row r0 + 16 * j: 16 * j * FT_ROW further)
        if (MODE == FT_PATCH) {
            const int total = my_tiles * p.chunks;
            int tile = mt0, ch = 0, s = 0, st = 0;
            uint32_t ph = 0, sph = 0;
            for (int a = 0; a < total; ++a) {
                if (!__all_sync(0xffffffffu, wait_bar(smem_u32(&sh->sa_full[st]), sph, abort_flag, p.status))) break;
                if (!__all_sync(0xffffffffu, wait_bar(smem_u32(&sh->a_empty[s]), ph ^ 1u, abort_flag, p.status))) break;
                // row r of the patch is position s0 + r; the staged rows start at a whole row of positions
                const int s0 = tile * FT_N - p.pad * (p.P + 1);
                const int row0 = s0 >= 0 ? fast_div(s0, p.div_p) : -1 - fast_div(-1 - s0, p.div_p);
                const uint32_t src = base + p.off_sa + (uint32_t)st * p.stage_a + (uint32_t)(s0 - row0 * p.P + r0) * 128u + (uint32_t)q * 16u;
                const uint32_t slot = base + (uint32_t)s * p.slot_a + my_quad;
                if (q < (ch == p.chunks - 1 ? 4 * p.ksteps_last : 8))       // (what the MMAs read; zeros past the last layer)
                    for (int rb = grp * 64; rb < p.prow; rb += 128) {
                        float4 v[4];
#pragma unroll
                        for (int j = 0; j < 4; ++j)
                            if (rb + r0 + 16 * j < p.prow) v[j] = ld_shared_v4(src + (uint32_t)(rb + 16 * j) * 128u);
#pragma unroll
                        for (int j = 0; j < 4; ++j)
                            if (rb + r0 + 16 * j < p.prow) store_split(slot + (uint32_t)((rb + 16 * j) * FT_ROW), p.plane_a, v[j]);
                    }
                fence_proxy_async_smem();               // planes visible to the tensor core
                __syncwarp();
                if (lane == 0) {
                    mbar_arrive(smem_u32(&sh->a_full[s]));
                    mbar_arrive(smem_u32(&sh->sa_empty[st]));
                }
                if (++s == p.ra) { s = 0; ph ^= 1u; }
                if (++st == p.sa) { st = 0; sph ^= 1u; }
                if (++ch == p.chunks) { ch = 0; tile += p.m_step; }
            }
        } else if (MODE == FT_FLAT) {
            const int total = my_tiles * p.chunks;
            int s = grp, st = grp;
            uint32_t sph = 0;
            for (int a = grp; a < total; a += 2) {
                if (!__all_sync(0xffffffffu, wait_bar(smem_u32(&sh->sa_full[st]), sph, abort_flag, p.status))) break;
                const uint32_t src = base + p.off_sa + (uint32_t)st * p.stage_a + (uint32_t)r0 * 128u + (uint32_t)q * 16u;
                float4 v[FT_NA];
#pragma unroll
                for (int j = 0; j < FT_NA; ++j) v[j] = ld_shared_v4(src + (uint32_t)(16 * 128 * j));
                if (!wait_done(a - p.ra)) break;
                const uint32_t slot = base + (uint32_t)s * p.slot_a + my_quad;
#pragma unroll
                for (int j = 0; j < FT_NA; ++j) store_split(slot + (uint32_t)(16 * j * FT_ROW), p.plane_a, v[j]);
                fence_proxy_async_smem();               // planes visible to the tensor core
                __syncwarp();
                if (lane == 0) {
                    mbar_arrive(smem_u32(&sh->a_full[s]));
                    mbar_arrive(smem_u32(&sh->sa_empty[st]));
                }
                s += 2;
                if (s >= p.ra) s -= p.ra;
                st += 2;
                if (st >= p.sa) { st -= p.sa; sph ^= 1u; }
            }
        } else {
            // steps = (tile, block of layers); both groups stage a step's box, one step ahead, and take its chunks in turn
            const int steps = my_tiles * p.nb;
            int f_tile = mt0, f_blk = 0;
            auto fill = [&](int step) {
                const uint32_t dst0 = base + p.off_sa + (uint32_t)(step & 1) * p.stage_a;
                const int t = fast_div(f_tile, p.div_tw), tx = f_tile - t * p.tiles_w, img = fast_div(t, p.div_th), ty = t - img * p.tiles_h;
                const int oh0 = ty * p.bh, ow0 = tx << p.bw_shift, c0 = f_blk * p.cb;
                const int nf = p.rc * p.cb;
                const bool dense = p.nb == 1 && p.S <= p.K;         // a box row is one run of floats
                for (int jr = warp; jr < p.rh; jr += 8) {
                    const int ih = p.S <= p.K ? oh0 * p.S - p.pad + jr : (oh0 + jr / p.K) * p.S - p.pad + jr % p.K;
                    const bool row_in = (unsigned)ih < (unsigned)p.H;
                    const float* row = p.in + ((size_t)img * p.H + (row_in ? ih : 0)) * p.W * p.Cin;
                    const uint32_t dst = dst0 + (uint32_t)(jr * p.pitch) * 4u;
                    const int iw0 = ow0 * p.S - p.pad;
                    const int unit = p.box_vec ? 4 : 1;
                    for (int f = lane * unit; f < nf; f += 32 * unit) {
                        long long off;
                        bool in = row_in;
                        if (dense) {
                            off = (long long)iw0 * p.Cin + f;
                            in = in && off >= 0 && off < (long long)p.W * p.Cin;
                        } else {
                            const int jc = fast_div(f, p.div_cb), c = f - jc * p.cb;
                            const int iw = p.S <= p.K ? iw0 + jc : (ow0 + jc / p.K) * p.S - p.pad + jc % p.K;
                            off = (long long)iw * p.Cin + c0 + c;
                            in = in && (unsigned)iw < (unsigned)p.W && c0 + c < p.Cin;
                        }
                        if (p.box_vec) cp_async_16(dst + 4u * f, in ? row + off : p.in, in);
                        else cp_async_4(dst + 4u * f, in ? row + off : p.in, in);
                    }
                }
                cp_async_commit();
                if (++f_blk == p.nb) { f_blk = 0; f_tile += p.m_step; }
            };
            uint32_t rowoff[FT_NA];
#pragma unroll
            for (int j = 0; j < FT_NA; ++j) {
                const int r = r0 + 16 * j, ty = r >> p.bw_shift, tx = r & ((1 << p.bw_shift) - 1);
                rowoff[j] = (uint32_t)(ty * p.stepb * p.pitch + tx * p.stepb * p.cb) * 4u;
            }
            chain_wait();
            if (steps > 0) fill(0);
            bool ok = true;                             // (a group that gives up still takes part in the barriers)
            int a = 0, s = 0;                           // chunk of the CTA's sequence, its slot
            for (int step = 0; step < steps; ++step) {
                asm volatile("cp.async.wait_group 0;" ::: "memory");
                bar_sync(1, 2 * FT_GT);                 // box filled by all; all have read the box of the step before
                if (step + 1 < steps) fill(step + 1);
                const uint32_t box = base + p.off_sa + (uint32_t)(step & 1) * p.stage_a;
                for (int ch = 0; ch < p.cpb; ++ch, ++a) {
                    if ((a & 1) == grp && ok) {
                        const int k = ch * FT_BK + 4 * q;
                        float4 v[FT_NA];
                        if (p.box_vec) {
                            const uint32_t o = box + (uint32_t)tbl[k].x * 4u;
#pragma unroll
                            for (int j = 0; j < FT_NA; ++j) v[j] = ld_shared_v4(o + rowoff[j]);
                        } else {
                            const uint32_t o0 = box + (uint32_t)tbl[k].x * 4u, o1 = box + (uint32_t)tbl[k + 1].x * 4u;
                            const uint32_t o2 = box + (uint32_t)tbl[k + 2].x * 4u, o3 = box + (uint32_t)tbl[k + 3].x * 4u;
#pragma unroll
                            for (int j = 0; j < FT_NA; ++j)
                                v[j] = make_float4(ld_shared_f32(o0 + rowoff[j]), ld_shared_f32(o1 + rowoff[j]), ld_shared_f32(o2 + rowoff[j]),
                                                   ld_shared_f32(o3 + rowoff[j]));
                        }
                        ok = wait_done(a - p.ra);
                        if (ok) {
                            const uint32_t slot = base + (uint32_t)s * p.slot_a + my_quad;
#pragma unroll
                            for (int j = 0; j < FT_NA; ++j) store_split(slot + (uint32_t)(16 * j * FT_ROW), p.plane_a, v[j]);
                            fence_proxy_async_smem();   // planes visible to the tensor core
                            __syncwarp();
                            if (lane == 0) mbar_arrive(smem_u32(&sh->a_full[s]));
                        }
                    }
                    if (++s == p.ra) s = 0;
                }
            }
        }
    } else if (warp < FT_W_EPI) {
        // ------------------------------------------------------------------ kernels: output layer n0 + row per thread
        asm volatile("setmaxnreg.dec.sync.aligned.u32 64;");
        const int quad = warp & 3, grp = (warp - FT_W_KER) >> 2, row = quad * 32 + lane;
        const uint32_t ta = tmem_base + ((uint32_t)(quad * 32) << 16) + FT_COL_W + (uint32_t)grp * FT_W_COLS;
        const int units = p.chunks * p.taps;
        const int total = p.kres ? units : my_tiles * units;
        // copies where the kernels' rows are no TMA tensor (BOX): lane -> reduction element, 32 rows per warp
        auto copy_rows = [&](int unit, uint32_t dst) {
            const int blk = unit / p.cpb;
            const int2 e = tbl[(unit - blk * p.cpb) * FT_BK + lane];
            const int off = e.y + blk * p.cb;
            const bool in = e.y >= 0 && e.y % p.Cin + blk * p.cb < p.Cin;
            const float* src = p.w + (size_t)(n0 + quad * 32) * p.Kdim + off;
            dst += (uint32_t)(quad * 32) * 128u + ((uint32_t)lane & 3u) * 4u;
            for (int i = 0; i < 32; ++i) {
                const bool ok = in && quad * 32 + i < n_live;
                cp_async_4(dst + (uint32_t)i * 128u + (((uint32_t)lane >> 2) ^ ((uint32_t)i & 7u)) * 16u, ok ? src + (size_t)i * p.Kdim : p.w, ok);
            }
        };
        const uint32_t boxes = base + p.off_sb + (uint32_t)grp * (2u * 128u * 128u);      // FT_W_COPIES: this group's two slots
        const uint32_t piece = (uint32_t)p.wrows * 16u;         // FT_W_PACKED: four packed pairs of every row
        const uint32_t unit_bytes = (p.khalf ? 6u : 12u) * piece;
        if (p.wsrc == FT_W_PACKED) {
            // quads of four reduction elements, consecutive threads on consecutive quads of a row, four in flight
            if (!p.early) chain_wait();
            const int ktid = tid - FT_W_KER * 32, qs = p.khalf ? 2 : 3, qn = 1 << qs;
            const int pieces = units * p.wrows * qn;
            for (int i0 = ktid; i0 < pieces; i0 += 4 * 2 * FT_GT) {
                float4 v[4];
                uint32_t dst[4];
#pragma unroll
                for (int e = 0; e < 4; ++e) {
                    const int i = i0 + e * 2 * FT_GT;
                    const int q = i & (qn - 1), ur = i >> qs, u = fast_div(ur, p.div_wrows), r = ur - u * p.wrows;
                    const int ch = fast_div(u, p.div_taps), tap = u - ch * p.taps;
                    v[e] = make_float4(0.f, 0.f, 0.f, 0.f);
                    const bool in = i < pieces && r < n_live;
                    const float* src = p.w + (size_t)(n0 + (in ? r : 0)) * p.Kdim;
                    if (MODE == FT_BOX) {
                        const int blk = u / p.cpb;
                        const int2* tb = tbl + (u - blk * p.cpb) * FT_BK + 4 * q;
                        auto at = [&](int2 k) {
                            return in && k.y >= 0 && (p.nb == 1 || k.y % p.Cin + blk * p.cb < p.Cin) ? __ldg(src + k.y + blk * p.cb) : 0.f;
                        };
                        if (i < pieces) v[e] = make_float4(at(tb[0]), at(tb[1]), at(tb[2]), at(tb[3]));
                    } else if (in && ch * FT_BK + 4 * q < p.Cin)
                        v[e] = __ldg(reinterpret_cast<const float4*>(src + (size_t)tap * p.Cin + ch * FT_BK + 4 * q));
                    dst[e] = base + p.off_sb + (uint32_t)u * unit_bytes + (uint32_t)(q >> 1) * piece + (uint32_t)r * 16u + ((uint32_t)q & 1u) * 8u;
                }
#pragma unroll
                for (int e = 0; e < 4; ++e)
                    if (i0 + e * 2 * FT_GT < pieces) store_split(dst[e], (p.khalf ? 2u : 4u) * piece, v[e]);
            }
            bar_sync(2, 2 * FT_GT);
        } else if (MODE == FT_BOX && p.wsrc == FT_W_COPIES) {
            if (!p.early) chain_wait();
            if (grp < total) copy_rows(grp % units, boxes);
            cp_async_commit();
        }
        bool ok = true;
        const bool idle = p.wsrc == FT_W_PACKED && quad * 32 >= p.wrows;                          // no rows to give: whatever is in these lanes of TMEM is never read
        int st = grp, unit = grp % units, sl = 0;       // box slot, unit of the tile
        uint32_t sph = 0;
        if (p.sb && st >= p.sb) { st -= p.sb; sph ^= 1u; }
        for (int u = grp; u < total; u += 2) {
            uint32_t h[16], m[16], l[16];
            int next_unit = unit + 2;
            while (next_unit >= units) next_unit -= units;
            if (p.wsrc == FT_W_PACKED) {
                if (!idle) {
                    const uint32_t src = base + p.off_sb + (uint32_t)unit * unit_bytes + (uint32_t)row * 16u, pl = (p.khalf ? 2u : 4u) * piece;
#pragma unroll
                    for (int i = 0; i < 4; ++i)
                        if (i < 2 || !p.khalf) {
                            ld_shared_u4(src + i * piece, &h[4 * i]);
                            ld_shared_u4(src + pl + i * piece, &m[4 * i]);
                            ld_shared_u4(src + 2u * pl + i * piece, &l[4 * i]);
                        }
                }
            } else {
                uint32_t src;
                if (MODE == FT_BOX && p.wsrc == FT_W_COPIES) {
                    asm volatile("cp.async.wait_group 0;" ::: "memory");
                    bar_sync(2 + grp, FT_GT);           // this unit's rows are here, the other slot has been read
                    if (u + 2 < total) copy_rows(next_unit, boxes + (uint32_t)(sl ^ 1) * (128u * 128u));
                    cp_async_commit();
                    src = boxes + (uint32_t)sl * (128u * 128u) + (uint32_t)row * 128u;
                    sl ^= 1;
                } else {
                    // An odd number of slots: the box before in this slot, unit u - sb's, was the other group's.  It has to be here first (its
                    // unit's MMAs are done), or this unit's, whose phase has the parity of the one before that, would look as if it
                    // were: where unit 1's box came later than unit 2's and unit 0's MMAs, unit 4 took its slot and gave it back twice.
                    if ((p.sb & 1) && !wait_done(u - p.sb)) break;
                    if (!__all_sync(0xffffffffu, wait_bar(smem_u32(&sh->sb_full[st]), sph, abort_flag, p.status))) break;
                    src = base + p.off_sb + (uint32_t)st * (128u * 128u) + (uint32_t)row * 128u;
                }
#pragma unroll
                for (int i = 0; i < 8; ++i) {
                    const float4 v = ld_shared_v4(src + (((uint32_t)i ^ ((uint32_t)row & 7u)) << 4));
                    split_pair(v.x, v.y, h[2 * i], m[2 * i], l[2 * i]);
                    split_pair(v.z, v.w, h[2 * i + 1], m[2 * i + 1], l[2 * i + 1]);
                }
                if (p.wsrc == FT_W_BOXES) {
                    __syncwarp();
                    if (lane == 0) mbar_arrive(smem_u32(&sh->sb_empty[st]));
                    st += 2;
                    while (st >= p.sb) { st -= p.sb; sph ^= 1u; }
                }
            }
            if (ok) ok = wait_done(u - FT_KSLOTS);
            if (ok) {
                tc_fence_after();
                if (idle) {
                } else if (p.khalf) {
                    tmem_st_x8(ta, h);
                    tmem_st_x8(ta + 16u, m);
                    tmem_st_x8(ta + 32u, l);
                } else {
                    tmem_st_x16(ta, h);
                    tmem_st_x16(ta + 16u, m);
                    tmem_st_x16(ta + 32u, l);
                }
                tmem_st_wait();
                tc_fence_before();
                __syncwarp();
                if (lane == 0) mbar_arrive(smem_u32(&sh->k_full[grp]));
            } else if (MODE != FT_BOX || p.wsrc != FT_W_COPIES) break;      // (with the copies the warps meet at a barrier in every turn)
            unit = next_unit;
        }
        if (MODE == FT_BOX) asm volatile("cp.async.wait_all;" ::: "memory");
    } else if (warp < FT_W_TMAX) {
        // -------------------------------------------------------------------------- epilogue
        asm volatile("setmaxnreg.inc.sync.aligned.u32 104;");
        const int quad = warp & 3, half = (warp - FT_W_EPI) >> 2;
        const uint32_t ta = tmem_base + ((uint32_t)(quad * 32) << 16) + (uint32_t)(half * 64);
        const int nseg = (p.chunks * p.taps + p.seg - 1) / p.seg;
        const int nw = n0 + quad * 32;                  // first output layer of this warp
        const int wl = n_live - quad * 32 < 32 ? n_live - quad * 32 : 32;       // output layers of this warp
        const bool vec = p.vec_store && wl % 4 == 0;
        float* out_w = p.out + p.out_c_offset + nw;
        const uint32_t stg0 = base + p.off_epi + (uint32_t)(quad * 2 + half) * (MODE != FT_PATCH && p.tstore ? (uint32_t)p.tstore * 128u : 2048u);
        if (!p.early) chain_wait();
        const float bias = lane < wl ? __ldg(p.bias + nw + lane) : 0.f;
        const float least = p.relu ? 0.f : bias != bias ? bias : -INFINITY;     // (fmaxf drops a NaN that only one operand has)
        // 16 staged pixels -> memory; lane l of mc has the output pixel of staged row l - first
        auto copy_out = [&](uint32_t stg, int mc, int first) {
            const int l4 = 4 * (lane & 7);
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                const float4 v = ld_shared_v4(stg + (uint32_t)(512 * i + 16 * lane));
                int m = __shfl_sync(0xffffffffu, mc, first + 4 * i + (lane >> 3));
                if (l4 >= wl || !sqn_dbg_ok(m < p.M && p.out_c_offset + nw + l4 < p.out_c_total, p.status)) m = -1;
                float* dst = out_w + (size_t)m * p.out_c_total + l4;
                if (vec) {
                    if (m >= 0) *reinterpret_cast<float4*>(dst) = v;
                } else if (m >= 0) {
                    dst[0] = v.x;
                    if (l4 + 1 < wl) dst[1] = v.y;
                    if (l4 + 2 < wl) dst[2] = v.z;
                    if (l4 + 3 < wl) dst[3] = v.w;
                }
            }
        };
        chain_wait();
        // output pixel of column c of a tile, -1: none
        auto pixel_of = [&](int tile, int c) {
            if (MODE == FT_PATCH) {
                const int pos = tile * FT_N + c;
                const int img = fast_div(pos, p.div_pos), r = pos - img * p.HP * p.P;
                const int y = fast_div(r, p.div_p), x = r - y * p.P;
                return img < p.N && y < p.OH && x < p.OW ? img * p.OHW + y * p.OW + x : -1;
            }
            if (MODE == FT_BOX) {
                const int tt = fast_div(tile, p.div_tw), tx = tile - tt * p.tiles_w, img = fast_div(tt, p.div_th), ty = tt - img * p.tiles_h;
                const int y = ty * p.bh + (c >> p.bw_shift), x = (tx << p.bw_shift) + (c & ((1 << p.bw_shift) - 1));
                return y < p.OH && x < p.OW ? img * p.OHW + y * p.OW + x : -1;
            }
            return tile * FT_N + c < p.M ? tile * FT_N + c : -1;
        };
        bool ok = quad < live_quads;                    // (warps without output layers are not counted by the barriers)
        int b = 0, first_unit = 0;
        const int units = p.chunks * p.taps;
        for (int t = 0; t < my_tiles && ok; ++t, first_unit += units) {
            float acc[64];
            // output pixels of columns lane and lane + 32 of this warp's half
            const int mc0 = pixel_of(mt0 + t * p.m_step, half * 64 + lane), mc1 = pixel_of(mt0 + t * p.m_step, half * 64 + 32 + lane);
#pragma unroll
            for (int c = 0; c < 64; ++c) acc[c] = 0.f;
            // the segments, and with the last of them the corrections, which are read first: the next tile waits for them
            for (int i = 0; i <= nseg; ++i) {
                const bool corr = i == nseg - 1;
                if (i < nseg) {
                    ok = wait_done(first_unit + (corr ? units : (i + 1) * p.seg) - 1);
                    if (!ok) break;
                    tc_fence_after();
                }
                const uint64_t cut = corr ? (uint64_t)__float_as_uint(FT_CUT) * 0x100000001ull : 0ull;      // (one copy of the unrolled code below: two of them spill)
                const uint32_t src = ta + (corr ? FT_COL_GX : (uint32_t)(b * FT_N));
#pragma unroll
                for (int c = 0; c < 64; c += 16) {
                    uint32_t v[16];
                    tmem_ld_x16(src + c, v);
                    tmem_ld_wait();
#pragma unroll
                    for (int j = 0; j < 16; j += 2) add_cut2(acc[c + j], acc[c + j + 1], cut, v[j], v[j + 1]);
                }
                tc_fence_before();
                __syncwarp();
                if (lane == 0) mbar_arrive(smem_u32(corr ? &sh->gx_empty : &sh->seg_empty[b]));
                if (!corr) b ^= 1;
            }
            if (!ok) break;
            // bias and ReLU here, where a thread has one layer and 64 independent pixels, then 16 pixels at a time through a
            // staging tile (a pixel's 32 layers are a row) and in 16-byte pieces, eight lanes per pixel, to memory; FLAT and BOX, whose
            // pixels are consecutive or boxes of the map: 16, 32 or 64 pixels, then a TMA store, which leaves out what lies outside the map
            // (BOX: conv1 at batch 256 1021 -> 975 us).  Only two warps per 32 layers have rows to store, so
            // the length of this chain is a tile's time where the reduction is short (fire2's 1x1 expand at batch 256 with
            // bias and ReLU after the staging tile and no TMA 107 us, so 80; a bulk copy per pixel instead of the 16-byte
            // pieces: fire2's expand-3x3 310 us instead of 230, conv1 1358 instead of 1011)
            float nan = 0.f;                            // 0 as long as all outputs are finite
#pragma unroll
            for (int c0 = 0; c0 < 64; c0 += 16) {
                // (TMA: a staging tile of that many pixels, free again when the store before has read it)
                const uint32_t stg = stg0 + (MODE != FT_PATCH && p.tstore ? (uint32_t)(c0 & (p.tstore - 1)) * 128u : 0u);
                if (MODE != FT_PATCH && lane == 0 && p.tstore && (c0 & (p.tstore - 1)) == 0) tma_store_wait_read();
                __syncwarp();
#pragma unroll
                for (int j = 0; j < 16; ++j) {
                    nan = fmaf(acc[c0 + j], 0.f, nan);
                    asm volatile("st.shared.f32 [%0], %1;" ::"r"(stg + (uint32_t)(128 * j + 4 * lane)), "f"(fmaxf(fmaf(acc[c0 + j], SPLIT_UNSCALE, bias), least)) : "memory");
                }
                if (MODE != FT_PATCH && p.tstore) {
                    if (((c0 + 16) & (p.tstore - 1)) == 0) {
                        fence_proxy_async_smem();
                        __syncwarp();
                        if (lane == 0) {
                            const int c = half * 64 + c0 + 16 - p.tstore, tile = mt0 + t * p.m_step;
                            if (MODE == FT_FLAT) {
                                if (tile * FT_N + c < p.M) tma_store_2d(&tmO, stg0, nw, tile * FT_N + c);
                            } else {
                                const int tt = fast_div(tile, p.div_tw), tx = tile - tt * p.tiles_w, img = fast_div(tt, p.div_th), ty = tt - img * p.tiles_h;
                                const int y = ty * p.bh + (c >> p.bw_shift), x = (tx << p.bw_shift) + (c & ((1 << p.bw_shift) - 1));
                                if (y < p.OH && x < p.OW) tma_store_4d(&tmO, stg0, nw, x, y, img);
                            }
                            tma_store_commit();
                        }
                    }
                } else {
                    __syncwarp();
                    copy_out(stg, c0 & 32 ? mc1 : mc0, c0 & 16);
                }
            }
            if (__any_sync(0xffffffffu, lane < wl && nan != 0.f)) {      // something was not finite: this warp's outputs with fp32 multiply-adds
                if (MODE != FT_PATCH && p.tstore && lane == 0) tma_store_wait_all();
                __syncwarp();
                float ws = 0.f;
                for (int c = -1; c < 64; ++c) {
                    const int m = c < 0 ? -1 : pixel_of(mt0 + t * p.m_step, half * 64 + c);
                    if (m < 0 && c >= 0) continue;
                    const float v = redo_output(p, m, nw + lane, ws);
                    if (c < 0) ws = v;
                    else if (lane < wl) out_w[(size_t)m * p.out_c_total + lane] = v;
                }
            }
        }
        if (MODE != FT_PATCH && p.tstore && lane == 0) tma_store_wait_all();
    } else {
        asm volatile("setmaxnreg.dec.sync.aligned.u32 40;");       // (of 28 x 32 x 72 registers: 104 for the epilogue, 64 for the groups that split)
        if (warp == FT_W_MMA) {
            // -------------------------------------------------------------------- MMA issuer
            // This warp's own instructions are what a unit takes at least (a barrier that is ready cost 150 to 350 clocks, a commit
            // 120, in all 1800 clocks a unit against 830 of MMAs): so the barriers of a unit are tried together, and one
            // commit serves all who wait for it.
            const uint32_t hi = (uint32_t)(make_kmajor_desc(0, FT_ROW, 8 * FT_ROW) >> 32);
            const uint32_t idesc = make_idesc_bf16(128, FT_N);
            const uint32_t PX = p.plane_a >> 4;             // plane pitch in 16-byte units
            auto desc = [&](uint32_t a16) { return ((uint64_t)hi << 32) | (uint64_t)(a16 | 0x10000u); };
            const uint32_t a_full = smem_u32(sh->a_full), k_full = smem_u32(sh->k_full), seg_empty = smem_u32(sh->seg_empty);
            const uint32_t gx = tmem_base + FT_COL_GX;
            const int units = p.chunks * p.taps, seg = p.seg;
            bool ok = true;
            uint32_t s = 0, ks = 0, b = 0, g = 0;
            uint32_t ph = 0, kph = 0, bph = 1, gph = 1;
            if (MODE == FT_BOX && units > 2) {
                // The last three MMAs of a unit go out behind a look at the next unit's barriers, so that the tensor pipe has work
                // meanwhile (it holds some four MMAs): conv1 at batch 256 1056 -> 1021 us.  (Not so with a patch: fire4's expand-3x3 368
                // -> 392; with one or two units to a tile fire4's expand-1x1 90 -> 94, 8 -> 323 2x2/2 13.5 -> 13.9; flat reductions of
                // more units gain 3 %, less than those lose.)
                const int total = my_tiles * units;
                int u = 0, in_seg = 0;
                bool ready = false;
                for (int i = 0; i < total; ++i) {
                    if (!ready) {
                        ok = wait_bar(a_full + 8u * s, ph, abort_flag, p.status);
                        ok = ok && (in_seg != 0 || wait_bar(seg_empty + 8u * b, bph, abort_flag, p.status));
                        ok = __all_sync(0xffffffffu, ok && wait_bar(k_full + 8u * ks, kph, abort_flag, p.status));
                        if (!ok) break;
                    }
                    tc_fence_after();
                    const uint32_t g0 = tmem_base + b * FT_N, w = tmem_base + FT_COL_W + ks * FT_W_COLS;
                    const uint64_t d0 = desc((base + s * p.slot_a) >> 4);       // the first plane; the others PX and 2 * PX further
                    const bool two = u != units - 1 || p.ksteps_last == 2;
                    if (elect_one()) {
                        mma_bf16_ts(g0, w, d0, idesc, in_seg ? 1u : 0u);
                        if (two) mma_bf16_ts(g0, w + 8u, d0 + 2u, idesc, 1u);
                    }
                    __syncwarp();
                    if (u == 0) {                           // the corrections of the tile before have to be read first
                        ok = __all_sync(0xffffffffu, wait_bar(smem_u32(&sh->gx_empty), gph, abort_flag, p.status));
                        gph ^= 1u;
                        if (!ok) break;
                        tc_fence_after();
                    }
                    if (elect_one()) {
                        mma_bf16_ts(gx, w, d0 + PX, idesc, u ? 1u : 0u);            // w0 x1
                        mma_bf16_ts(gx, w, d0 + 2u * PX, idesc, 1u);                // w0 x2
                        if (two) {
                            mma_bf16_ts(gx, w + 16u, d0, idesc, 1u);                // w1 x0
                            mma_bf16_ts(gx, w + 16u, d0 + PX, idesc, 1u);           // w1 x1
                            mma_bf16_ts(gx, w + 32u, d0, idesc, 1u);                // w2 x0
                            mma_bf16_ts(gx, w + 8u, d0 + PX + 2u, idesc, 1u);
                            mma_bf16_ts(gx, w + 8u, d0 + 2u * PX + 2u, idesc, 1u);
                        }
                    }
                    __syncwarp();
                    const uint32_t wl = two ? w + 8u : w;
                    const uint64_t dl = two ? d0 + 2u : d0;
                    ks ^= 1u; kph ^= ks ^ 1u;
                    if (u == units - 1 || in_seg == seg - 1) {
                        in_seg = 0;
                        b ^= 1u; bph ^= b ^ 1u;
                    } else ++in_seg;
                    if (++u == units) u = 0;
                    if (++s == (uint32_t)p.ra) { s = 0; ph ^= 1u; }
                    ready = false;
                    if (i + 1 < total) {
                        ready = mbar_test_wait(a_full + 8u * s, ph);
                        ready &= in_seg != 0 || mbar_test_wait(seg_empty + 8u * b, bph);
                        ready &= mbar_test_wait(k_full + 8u * ks, kph);
                        ready = __all_sync(0xffffffffu, ready);
                    }
                    if (elect_one()) {
                        mma_bf16_ts(gx, wl + 16u, dl, idesc, 1u);
                        mma_bf16_ts(gx, wl + 16u, dl + PX, idesc, 1u);
                        mma_bf16_ts(gx, wl + 32u, dl, idesc, 1u);
                        mma_commit(done + 8u * ((uint32_t)i & 3u));
                    }
                    __syncwarp();
                }
            } else
            for (int t = 0; t < my_tiles && ok; ++t) {
                int in_seg = 0, u = 0;
                for (int ch = 0; ch < p.chunks && ok; ++ch) {
                    uint32_t lo = (base + s * p.slot_a) >> 4;
                    const bool two = ch != p.chunks - 1 || p.ksteps_last == 2;
                    int kw = 0;
                    for (int tap = 0; tap < p.taps; ++tap, ++u, ++g) {
                        const uint32_t af = a_full + 8u * s, se = seg_empty + 8u * b, kf = k_full + 8u * ks;
                        const bool need_a = tap == 0, need_s = in_seg == 0, need_k = !p.kres || t == 0;
                        bool ready = !need_a || mbar_try_wait(af, ph);
                        ready &= !need_s || mbar_try_wait(se, bph);
                        ready &= !need_k || mbar_try_wait(kf, kph);
                        if (!__all_sync(0xffffffffu, ready)) {
                            ok = !need_a || wait_bar(af, ph, abort_flag, p.status);
                            ok = ok && (!need_s || wait_bar(se, bph, abort_flag, p.status));
                            ok = __all_sync(0xffffffffu, ok && (!need_k || wait_bar(kf, kph, abort_flag, p.status)));
                            if (!ok) break;
                        }
                        tc_fence_after();
                        const uint32_t g0 = tmem_base + b * FT_N, w = tmem_base + FT_COL_W + ks * FT_W_COLS;
                        const uint64_t d0 = desc(lo), d1 = d0 + PX, d2 = d1 + PX;       // the planes
                        const bool seg_end = u == units - 1 || in_seg == seg - 1;
                        if (u == 0) {                       // the corrections of the tile before have to be read first
                            if (elect_one()) {
                                mma_bf16_ts(g0, w, d0, idesc, 0u);
                                if (two) mma_bf16_ts(g0, w + 8u, d0 + 2u, idesc, 1u);
                            }
                            __syncwarp();
                            ok = __all_sync(0xffffffffu, wait_bar(smem_u32(&sh->gx_empty), gph, abort_flag, p.status));
                            gph ^= 1u;
                            if (!ok) break;
                            tc_fence_after();
                        }
                        if (elect_one()) {
                            if (u) {
                                mma_bf16_ts(g0, w, d0, idesc, in_seg ? 1u : 0u);
                                if (two) mma_bf16_ts(g0, w + 8u, d0 + 2u, idesc, 1u);
                            }
                            mma_bf16_ts(gx, w, d1, idesc, u ? 1u : 0u);             // w0 x1
                            mma_bf16_ts(gx, w, d2, idesc, 1u);                      // w0 x2
                            mma_bf16_ts(gx, w + 16u, d0, idesc, 1u);                // w1 x0
                            mma_bf16_ts(gx, w + 16u, d1, idesc, 1u);                // w1 x1
                            mma_bf16_ts(gx, w + 32u, d0, idesc, 1u);                // w2 x0
                            if (two) {
                                mma_bf16_ts(gx, w + 8u, d1 + 2u, idesc, 1u);
                                mma_bf16_ts(gx, w + 8u, d2 + 2u, idesc, 1u);
                                mma_bf16_ts(gx, w + 24u, d0 + 2u, idesc, 1u);
                                mma_bf16_ts(gx, w + 24u, d1 + 2u, idesc, 1u);
                                mma_bf16_ts(gx, w + 40u, d0 + 2u, idesc, 1u);
                            }
                            mma_commit(done + 8u * (g & 3u));
                            if (MODE == FT_PATCH && tap == p.taps - 1) mma_commit(smem_u32(&sh->a_empty[s]));
                        }
                        __syncwarp();
                        if (p.kres) { if (++ks == (uint32_t)units) ks = 0; }    // (unit u of a tile stays in slot u)
                        else { ks ^= 1u; kph ^= ks ^ 1u; }
                        if (seg_end) {
                            in_seg = 0;
                            b ^= 1u; bph ^= b ^ 1u;
                        } else ++in_seg;
                        if (MODE == FT_PATCH) {             // the next tap starts a row of the patch further, a kernel row P rows
                            lo += FT_ROW >> 4;
                            if (++kw == p.K) { kw = 0; lo += (uint32_t)(p.P - p.K) * (FT_ROW >> 4); }
                        }
                    }
                    if (++s == (uint32_t)p.ra) { s = 0; ph ^= 1u; }
                }
            }
        } else if ((warp == FT_W_TMAX || warp == FT_W_TMAW) && lane == 0) {
            // -------------------------------------------------------------------- TMA producers
            bool ok = true;
            int st = 0, issued = 0;
            uint32_t ph = 0;
            const bool px = warp == FT_W_TMAX;
            const int slots = px ? p.sa : p.wsrc == FT_W_BOXES ? p.sb : 0;
            unsigned long long *full = px ? sh->sa_full : sh->sb_full, *empty = px ? sh->sa_empty : sh->sb_empty;
            auto claim = [&](uint32_t bytes) {
                ok = wait_bar(smem_u32(&empty[st]), ph ^ 1u, abort_flag, p.status);
                if (ok) mbar_arrive_expect_tx(smem_u32(&full[st]), bytes);
                return ok;
            };
            auto next = [&]() {
                ++issued;
                if (++st == slots) { st = 0; ph ^= 1u; }
            };
            if (px && slots) {
                chain_wait();
                const uint32_t rows_bytes = (uint32_t)p.P * 128u;
                for (int t = 0; t < my_tiles && ok; ++t) {
                    const int tile = mt0 + t * p.m_step;
                    if (MODE == FT_FLAT) {
                        for (int ch = 0; ch < p.chunks; ++ch) {
                            if (!claim(FT_N * 128)) break;
                            tma_load_2d(base + p.off_sa + (uint32_t)st * p.stage_a, &tmX, smem_u32(&full[st]), ch * FT_BK, tile * FT_N);
                            next();
                        }
                    } else {
                        // one box per row of positions: what lies outside the map (the padding) is filled with zeros
                        const int s0 = tile * FT_N - p.pad * (p.P + 1);
                        const int row0 = s0 >= 0 ? fast_div(s0, p.div_p) : -1 - fast_div(-1 - s0, p.div_p);
                        const int row1 = fast_div(s0 + p.prow - 1, p.div_p);
                        for (int ch = 0; ch < p.chunks; ++ch) {
                            if (!claim((uint32_t)(row1 - row0 + 1) * rows_bytes)) break;
                            int img = row0 >= 0 ? row0 / p.HP : 0, y = row0 - img * p.HP;
                            for (int r = row0; r <= row1; ++r) {
                                tma_load_5d(base + p.off_sa + (uint32_t)st * p.stage_a + (uint32_t)(r - row0) * rows_bytes, &tmX, smem_u32(&full[st]),
                                            ch * FT_BK, 0, y, img, 0);
                                if (++y == p.HP) { y = 0; ++img; }
                            }
                            next();
                        }
                    }
                }
            } else if (!px && slots) {
                if (!p.early) chain_wait();
                for (int t = 0; t < (p.kres ? 1 : my_tiles) && ok; ++t)
                    for (int ch = 0; ch < p.chunks && ok; ++ch)
                        for (int tap = 0; tap < p.taps; ++tap) {
                            if (!claim(128 * 128)) break;
                            tma_load_2d(base + p.off_sb + (uint32_t)st * (128u * 128u), &tmW, smem_u32(&full[st]), tap * p.Cin + ch * FT_BK, n0);
                            next();
                        }
            }
            if (!ok)        // give the boxes already issued a bounded chance to land before the CTA exits
                for (int pending = issued < slots ? issued : slots; pending > 0; --pending) {
                    if (st == 0) { st = slots; ph ^= 1u; }
                    --st;
                    const long long t0 = clock64();
                    while (!mbar_try_wait(smem_u32(&full[st]), ph)) {
                        if (clock64() - t0 > WAIT_LIMIT_CYCLES / 8) break;
                        __nanosleep(100);
                    }
                }
        }
    }

    tc_fence_before();
    __syncthreads();
    if (warp == FT_W_MMA) {
        __syncwarp();
        tc_fence_after();
        tmem_dealloc(tmem_base, 512);
    }
}

template <int MODE>
__global__ void __launch_bounds__(FT_THREADS, 1)
conv_f32_tc_kernel(const __grid_constant__ CUtensorMap tmX, const __grid_constant__ CUtensorMap tmW,
                   const __grid_constant__ CUtensorMap tmO, const __grid_constant__ F32TcParams p)
{
    conv_f32_tc_body<MODE>(tmX, tmW, tmO, p, (int)blockIdx.x);
}

// ------------------------------------------------------------------------------ host side
struct F32TcPlan {
    CUtensorMap x, w, o;
    F32TcParams p;
    size_t smem;
};

inline int ceil_div(long long a, long long b) { return (int)((a + b - 1) / b); }
inline size_t up1k(size_t v) { return (v + 1023) / 1024 * 1024; }

// Shared-memory layout; returns its size, 0 if it does not fit.
size_t layout(F32TcParams& p)
{
    const int units = p.chunks * p.taps;
    p.plane_a = (unsigned)up1k((size_t)p.prow * FT_ROW);
    p.slot_a = 3u * p.plane_a;
    // PATCH: the staged rows of a patch, of which the first and the last are not all needed
    p.stage_a = (unsigned)up1k(p.mode == FT_FLAT ? (size_t)FT_N * 128 : p.mode == FT_PATCH ? (size_t)((p.prow - 2) / p.P + 2) * p.P * 128
                                                                                           : (size_t)p.rh * p.pitch * 4);
    const size_t tbl = p.mode == FT_BOX ? up1k((size_t)p.cpb * FT_BK * 8) : 0;
    static_assert(sizeof(F32TcShared) <= 1024, "control block");
    // {pixel slots, pixel boxes, kernel boxes}: FLAT and BOX slots are taken in turn by two groups
    static const int flat[][3] = {{4, 4, 3}, {2, 4, 3}}, patch[][3] = {{2, 2, 3}, {2, 1, 3}, {2, 1, 2}, {1, 1, 2}}, box[][3] = {{4, 2, 3}, {2, 2, 3}};
    const int(*cand)[3] = p.mode == FT_FLAT ? flat : p.mode == FT_PATCH ? patch : box;
    const int n = p.mode == FT_PATCH ? 4 : 2, n_packed = 2;
    const int streamed = p.mode != FT_BOX || (p.nb == 1 && p.Kdim % 4 == 0) ? FT_W_BOXES : FT_W_COPIES;
    p.khalf = p.chunks == 1 && p.ksteps_last == 1 ? 1 : 0;
    p.wrows = (p.n_step + 31) / 32 * 32;
    p.div_wrows = make_div(p.wrows); p.div_taps = make_div(p.taps);
    for (int i = 0; i < n_packed + n; ++i) {
        const int* c = cand[i < n_packed ? i : i - n_packed];
        p.wsrc = i < n_packed ? FT_W_PACKED : streamed;
        p.ra = c[0];
        p.sa = c[1];
        p.sb = p.wsrc == FT_W_PACKED ? 0 : p.wsrc == FT_W_COPIES ? 4 : p.kres ? units : c[2];
        size_t cur = (size_t)p.ra * p.slot_a;
        p.off_sa = (unsigned)cur; cur += (size_t)p.sa * p.stage_a;
        p.off_sb = (unsigned)cur; cur += p.wsrc == FT_W_PACKED ? up1k((size_t)units * p.wrows * (p.khalf ? 96 : 192)) : (size_t)p.sb * 128 * 128;
        p.off_epi = (unsigned)cur; cur += p.tstore > 16 ? (size_t)2 * ((p.n_step + 31) / 32) * p.tstore * 128 : 8 * 2048;
        p.off_tbl = (unsigned)cur; cur += tbl;
        p.off_ctl = (unsigned)cur; cur += 1024;
        if (cur + 1024 > FT_SMEM_LIMIT) continue;
        if (p.mode == FT_BOX) p.sa = 0;                 // (no TMA boxes)
        return cur + 1024;
    }
    return 0;
}

// Microseconds this kernel takes: start and end of a launch, then per tile of the busiest CTA its epilogue and its units of 32
// (or 16) reduction elements.  FLAT and PATCH: fitted to SqueezeNet's layers at batch 1 .. 256 (500 random layers: 0.85 to 1.2
// of it in nine of ten).  BOX: the copies of a tile's windows, a thread's share one after the other (0.05 us each where a window
// row is one run of memory, else 0.1) and 0.4 us for every block of layers, and the kernels' split, once; fitted to 890 random
// layers with a stride or odd layer counts (0.9 to 1.15 of it in eight of ten, 1.7 at most; without these terms 1.0 to 6.5, and a
// 1x1/3 layer of 28 images, 151 -> 53 at 57 x 49, went here for 40 us in the place of 15).
float f32_tc_estimate(const F32TcParams& p)
{
    if (p.mode == FT_BOX) {
        const int copies = ceil_div(p.rh, 8) * ceil_div((long long)p.rc * p.cb, p.box_vec ? 128 : 32);
        const float unit = p.wsrc == FT_W_COPIES ? 1.24f : 0.8f, packed = p.wsrc == FT_W_PACKED ? (float)(p.chunks * p.wrows) / 128.f : 0.f;
        const float tile = 2.f + unit * (float)p.chunks + (float)p.nb * (0.4f + (p.nb == 1 && p.S <= p.K ? 0.047f : 0.1f) * (float)copies);
        return 3.5f + 1.5f * (p.khalf ? 0.5f : 1.f) * packed + (float)ceil_div(p.m_tiles, p.m_step) * ceil_div(p.grid, sm_count()) * tile;
    }
    const float unit = p.wsrc != FT_W_PACKED && p.mode != FT_PATCH ? 0.9f : p.khalf ? 0.45f : 0.63f;
    return 4.5f + (float)ceil_div(p.m_tiles, p.m_step) * ceil_div(p.grid, sm_count()) * (1.6f + unit * (float)(p.chunks * p.taps));
}

int build_f32_plan(const ConvDesc& d, F32TcPlan* plan)
{
    F32TcParams& p = plan->p;
    std::memset(plan, 0, sizeof(*plan));
    p.in = static_cast<const float*>(d.in);
    p.w = static_cast<const float*>(d.w);
    p.bias = d.bias;
    p.out = static_cast<float*>(d.out);
    p.status = device_status_word();
    const long long M = (long long)d.N * d.OH * d.OW;
    const long long Kdim = (long long)d.K * d.K * d.Cin;
    if (M <= 0 || M > 0x7fffffffLL - 512 || Kdim > 0x7fffffffLL - 64) return SQN_ERR_UNSUPPORTED;
    if ((long long)d.H * d.W * d.Cin > 0x7fffffffLL) return SQN_ERR_UNSUPPORTED;
    p.N = d.N; p.Cin = d.Cin; p.H = d.H; p.W = d.W; p.Cout = d.Cout; p.K = d.K; p.S = d.S; p.pad = d.pad;
    p.OH = d.OH; p.OW = d.OW; p.OHW = d.OH * d.OW;
    p.M = (int)M; p.Kdim = (int)Kdim;
    p.out_c_offset = d.out_c_offset; p.out_c_total = d.out_c_total; p.relu = d.relu;
    p.div_ohw = make_div(p.OHW); p.div_ow = make_div(p.OW);
    p.early = d.params_static;
    p.vec_store = d.out_c_offset % 4 == 0 && d.out_c_total % 4 == 0;
    const int sms = sm_count();
    p.n_tiles = ceil_div(d.Cout, 128);
    p.n_step = ceil_div(ceil_div(d.Cout, p.n_tiles), 32) * 32;
    p.n_tiles = ceil_div(d.Cout, p.n_step);

    const bool vec = d.Cin % 4 == 0;
    p.P = d.W + d.pad; p.HP = d.H + d.pad;
    const long long positions = (long long)d.N * p.HP * p.P;
    auto finish = [&](int span, long long pixels) {         // reduction per tap (or in all), and the tiles
        p.chunks = p.mode == FT_BOX ? p.nb * p.cpb : ceil_div(span, FT_BK);
        p.ksteps_last = span - (ceil_div(span, FT_BK) - 1) * FT_BK > 16 ? 2 : 1;
        if (p.mode == FT_BOX && p.nb > 1) p.ksteps_last = 2;
        p.seg = p.chunks == 1 && p.ksteps_last == 1 ? 2 : 1;      // 32 reduction elements
        p.kres = p.chunks * p.taps <= FT_KSLOTS ? 1 : 0;
        p.m_tiles = p.mode == FT_BOX ? d.N * p.tiles_h * p.tiles_w : ceil_div(pixels, FT_N);
        plan->smem = layout(p);
        return plan->smem != 0;
    };
    auto grid = [&](F32TcParams& q) {
        q.m_step = sms / q.n_tiles;
        if (q.m_step < 1) q.m_step = 1;
        if (q.m_step > q.m_tiles) q.m_step = q.m_tiles;
        q.grid = q.n_tiles * q.m_step;
    };
    bool found = false;
    p.taps = 1;
    if (vec && d.K == 1 && d.S == 1 && d.pad == 0) {
        p.mode = FT_FLAT;
        p.prow = FT_N;
        p.tstore = !p.vec_store || d.Cout % 4 != 0 ? 0 : p.n_step <= 64 ? 64 : 32;      // (TMA writes whole 16-byte pieces)
        found = finish(d.Cin, M);
    } else if (vec && d.K > 1 && d.S == 1 && d.pad < d.K && p.P <= 256 && positions < 0x7fffffffLL - 2 * FT_N - (long long)d.K * (p.P + 1)) {
        p.mode = FT_PATCH;
        p.prow = FT_N + (d.K - 1) * (p.P + 1);
        p.taps = d.K * d.K;
        p.div_pos = make_div(p.HP * p.P); p.div_p = make_div(p.P);
        found = finish(d.Cin, positions);
    }
    if (!found) {
        p.mode = FT_BOX;
        p.prow = FT_N;
        p.taps = 1;
        // tile shape with the fewest tiles (the smaller box on ties), layers per block as many as fit
        auto search = [&](int tstore, F32TcPlan* found) {
            long long best = -1;
            p.tstore = tstore;
            for (int sh = 7; sh >= 0; --sh) {
                const int bw = 1 << sh, bh = 128 >> sh;
                p.stepb = d.S < d.K ? d.S : d.K;
                p.rh = (bh - 1) * p.stepb + d.K; p.rc = (bw - 1) * p.stepb + d.K;
                p.bw_shift = sh; p.bh = bh;
                p.tiles_w = ceil_div(d.OW, bw); p.tiles_h = ceil_div(d.OH, bh);
                const long long tiles = (long long)p.tiles_w * p.tiles_h;
                if (tiles * d.N > 0x3fffffffLL) continue;
                p.div_tw = make_div(p.tiles_w); p.div_th = make_div(p.tiles_h);
                for (int cb = d.Cin; cb > 0; cb = cb > 32 ? 32 : cb / 2 / 4 * 4) {
                    if ((long long)d.K * d.K * cb > FT_TBL_MAX || (long long)p.rh * p.rc * cb * 4 > 64 * 1024) continue;
                    p.cb = cb;
                    p.nb = ceil_div(d.Cin, cb);
                    p.cpb = ceil_div((long long)d.K * d.K * cb, FT_BK);
                    p.pitch = (p.rc * cb + 3) / 4 * 4;
                    p.box_vec = vec && cb % 4 == 0 ? 1 : 0;
                    p.div_cb = make_div(cb);
                    const long long cost = tiles * 1000000 + (long long)p.rh * p.rc * cb;
                    if (best >= 0 && cost >= best) break;
                    if (!finish(d.K * d.K * cb, 0)) continue;
                    best = cost;
                    *found = *plan;
                    grid(found->p);
                    break;
                }
            }
            return best >= 0;
        };
        // TMA stores of 32 pixels need more staging than those of 16, which need no more than stores without TMA: other tiles, a poorer
        // source of the kernels or more blocks.  The better plan by its estimate, 32 pixels where they are equal (conv1 at batch 256
        // 970 us with two pixel slots and 32 pixels, 1008 with four and 16).  188 random layers, geometric mean, plain stores 1: this
        // 0.975, always 32 0.981, 16 ahead of a poorer plan 0.983.  18 -> 348 3x3/2 at 43 x 42, 48 images, 79 us with 16, 130 with 32 in
        // three blocks; 4 -> 164 7x7/2 at 56 x 53, 20 images, 21 with 32 and kernels by boxes, 28 with 16 and packed ones.
        const bool tma = p.vec_store && d.Cout % 4 == 0;
        F32TcPlan bp, other;
        const bool a = search(tma ? 32 : 0, &bp), b = tma && search(16, &other);
        if (!a && !b) return SQN_ERR_UNSUPPORTED;
        *plan = !a || (b && f32_tc_estimate(other.p) < f32_tc_estimate(bp.p)) ? other : bp;
        return SQN_OK;
    }
    grid(p);
    return SQN_OK;
}

int encode_f32_maps(const ConvDesc& d, F32TcPlan* plan)
{
    const F32TcParams& p = plan->p;
    if (p.mode == FT_FLAT) {
        // pixels as [pixel][layer], boxes of 128 pixels x 32 layers
        const cuuint64_t dims[2] = {(cuuint64_t)d.Cin, (cuuint64_t)p.M}, str[1] = {(cuuint64_t)d.Cin * 4};
        const cuuint32_t box[2] = {FT_BK, FT_N};
        if (!tmap_encode_f32(&plan->x, 2, d.in, dims, str, box, 0)) return SQN_ERR_CUDA;
    } else if (p.mode == FT_PATCH) {
        const cuuint64_t s1 = (cuuint64_t)d.Cin * 4;
        const cuuint64_t dims[5] = {(cuuint64_t)d.Cin, (cuuint64_t)d.W, (cuuint64_t)d.H, (cuuint64_t)d.N, 1};
        const cuuint64_t str[4] = {s1, s1 * d.W, s1 * d.W * d.H, s1 * d.W * d.H * d.N};
        const cuuint32_t box[5] = {FT_BK, (cuuint32_t)p.P, 1, 1, 1};
        if (!tmap_encode_f32(&plan->x, 5, d.in, dims, str, box, 0)) return SQN_ERR_CUDA;
    }
    if (p.tstore) {
        // this layer's slice of the output
        const cuuint64_t s1 = (cuuint64_t)d.out_c_total * 4;
        if (p.mode == FT_FLAT) {
            const cuuint64_t dims[2] = {(cuuint64_t)d.Cout, (cuuint64_t)p.M}, str[1] = {s1};
            const cuuint32_t box[2] = {32, (cuuint32_t)p.tstore};
            if (!tmap_encode_f32(&plan->o, 2, p.out + p.out_c_offset, dims, str, box, 0)) return SQN_ERR_CUDA;
        } else {
            const cuuint64_t dims[4] = {(cuuint64_t)d.Cout, (cuuint64_t)d.OW, (cuuint64_t)d.OH, (cuuint64_t)d.N};
            const cuuint64_t str[3] = {s1, s1 * d.OW, s1 * d.OW * d.OH};
            const cuuint32_t bw = 1u << p.bw_shift, w = bw < (cuuint32_t)p.tstore ? bw : (cuuint32_t)p.tstore;
            const cuuint32_t box[4] = {32, w, (cuuint32_t)p.tstore / w, 1};
            if (!tmap_encode_f32(&plan->o, 4, p.out + p.out_c_offset, dims, str, box, 0)) return SQN_ERR_CUDA;
        }
    }
    if (p.wsrc == FT_W_BOXES) {
        const cuuint64_t dims[2] = {(cuuint64_t)p.Kdim, (cuuint64_t)d.Cout}, str[1] = {(cuuint64_t)p.Kdim * 4};
        const cuuint32_t box[2] = {FT_BK, 128};
        if (!tmap_encode_f32(&plan->w, 2, d.w, dims, str, box, 128)) return SQN_ERR_CUDA;
    }
    return SQN_OK;
}

template <int MODE>
cudaError_t launch_mode(const F32TcPlan& plan, cudaStream_t stream)
{
    static SmemAttr attr;
    const cudaError_t arc = attr.allow((const void*)conv_f32_tc_kernel<MODE>, FT_SMEM_LIMIT);
    if (arc != cudaSuccess) return arc;
    return launch_chained(conv_f32_tc_kernel<MODE>, dim3((unsigned)plan.p.grid), dim3(FT_THREADS), plan.smem, stream, plan.x, plan.w, plan.o, plan.p);
}

}  // namespace

int launch_conv_f32_tc(const ConvDesc& d, float limit_us, cudaStream_t stream)
{
    F32TcPlan plan;
    const int rc = build_f32_plan(d, &plan);
    if (rc != SQN_OK) return rc;
    if (f32_tc_estimate(plan.p) > limit_us) return SQN_ERR_UNSUPPORTED;
    if (encode_f32_maps(d, &plan) != SQN_OK) return SQN_ERR_CUDA;
    const cudaError_t e = plan.p.mode == FT_FLAT ? launch_mode<FT_FLAT>(plan, stream)
                        : plan.p.mode == FT_PATCH ? launch_mode<FT_PATCH>(plan, stream) : launch_mode<FT_BOX>(plan, stream);
    if (e != cudaSuccess) return SQN_ERR_CUDA;
    const F32TcParams& p = plan.p;
    const bool stores = p.mode == FT_BOX && p.tstore;
    note_launch(stores ? "conv_f32_tc %s, kernels %s, %d %s%s, %d pixels per store" : "conv_f32_tc %s, kernels %s, %d %s%s",
                p.mode == FT_FLAT ? "flat" : p.mode == FT_PATCH ? "patch" : "box",
                p.wsrc == FT_W_PACKED ? "packed" : p.wsrc == FT_W_BOXES ? "by boxes" : "by copies", p.mode == FT_BOX ? p.nb : 1,
                p.mode == FT_BOX && p.nb > 1 ? "blocks" : "block", p.mode == FT_BOX && p.S > p.K ? ", apart" : "", p.tstore);
    return cudaGetLastError() == cudaSuccess ? SQN_OK : SQN_ERR_CUDA;
}

}  // namespace sqn
