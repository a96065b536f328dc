"""The exact path's tensor-core kernel (every fp32 operand as three bf16 numbers) against the oracle, at the sizes where its
tiles, chunks and dispatch branches end.  That a shape really runs on it, and in which variant, is asserted by name.

Bound per output, S = sum of |kernel * input| over the window: the products left out are below 2^-22 of the operands'
product; a segment of 32 products is cut to 24 bits in two steps of at most 2^-23 of what it holds, the segments are added
with rounded additions (2^-24 each), and so are corrections and bias."""
import numpy as np
import pytest

from oracle import ref
from paper_1611_07151_b200 import binding as B
from paper_1611_07151_b200 import synth
import gpu_util as G

pytestmark = pytest.mark.gpu
F32 = B.SQN_F32

# (N, Cin, Cout, H, K, S, pad), the variant that runs
SHAPES = [
    ((40, 128, 32, 55, 1, 1, 0), "flat, kernels packed"),           # a quarter of the MMA rows live
    ((11, 260, 130, 27, 1, 1, 0), "flat, kernels by boxes"),        # last chunk of 4, two columns of tiles, ragged everywhere
    ((3, 512, 1000, 13, 1, 1, 0), "flat, kernels by boxes"),        # eight columns of tiles
    ((24, 16, 64, 55, 3, 1, 1), "patch, kernels packed"),           # units of 16 reduction elements
    ((9, 48, 192, 27, 3, 1, 1), "patch, kernels by boxes"),         # last chunk of 16, 96 layers per column
    ((8, 64, 130, 33, 3, 1, 1), "patch, kernels by boxes"),
    ((6, 36, 70, 40, 5, 1, 2), "patch, kernels by boxes"),          # 5x5, chunk of 4
    ((4, 32, 64, 60, 3, 1, 0), "patch, kernels by boxes"),          # no padding
    ((6, 32, 96, 41, 2, 1, 1), "patch, kernels packed"),            # even kernel, output larger than the input
    ((5, 3, 96, 111, 7, 2, 0), "box, kernels packed, 1 block"),     # layers not a multiple of 4
    ((46, 8, 323, 31, 2, 2, 1), "box, kernels packed, 1 block"),    # ... a multiple of 4
    ((34, 16, 496, 50, 1, 2, 0), "box, kernels packed, 1 block, apart"),        # windows apart from one another
    ((42, 122, 124, 18, 1, 1, 0), "box, kernels packed, 4 blocks"),
    ((40, 124, 128, 58, 1, 2, 0), "box, kernels packed, 4 blocks, apart"),
    ((1, 64, 64, 300, 3, 1, 1), "box, kernels by boxes, 1 block"),  # rows too long for the patch
    ((30, 47, 308, 7, 2, 1, 1), "box, kernels by boxes, 1 block"),
    ((43, 24, 353, 26, 2, 3, 0), "box, kernels by boxes, 1 block, apart"),
    ((60, 11, 2, 38, 7, 2, 0), "box, kernels by copies, 1 block"),  # two output layers
    ((25, 95, 109, 60, 1, 2, 0), "box, kernels by copies, 1 block, apart"),
    ((16, 64, 128, 56, 3, 2, 1), "box, kernels by copies, 4 blocks"),           # 16-byte pieces
    ((23, 36, 304, 30, 2, 2, 0), "box, kernels by copies, 3 blocks"),           # ... the last block of 4 layers
    ((20, 77, 133, 21, 3, 1, 1), "box, kernels by copies, 3 blocks"),           # 4-byte pieces
    ((60, 206, 97, 25, 1, 2, 0), "box, kernels by copies, 7 blocks, apart"),
]

def bound(x, w, b, S, pad, K, C):
    z = np.zeros_like(b)
    terms = ref.conv2d(np.abs(x), np.abs(w), z, S=S, pad=pad, relu=False).astype(np.float64)
    return (2.0 ** -22 + 2 * 2.0 ** -23 + (K * K * C / 32 + 4) * 2.0 ** -24) * (terms + np.abs(b)[None, :, None, None])


@pytest.mark.parametrize("shape,variant", SHAPES, ids=["x".join(map(str, s)) for s, _ in SHAPES])
def test_tensor_core_kernel_within_rounding(shape, variant):
    N, C, M, H, K, S, pad = shape
    rng = np.random.default_rng(sum(shape))
    x = rng.standard_normal((N, C, H, H - 2)).astype(np.float32)
    w, b = synth.draw_conv_params(rng, C, M, K)
    exp = ref.conv2d(x, w, b, S=S, pad=pad, relu=False)
    got = G.gpu_conv(x, w, b, S, pad, False, F32, kernel="conv_f32_tc " + variant)
    assert got.shape == exp.shape
    assert (np.abs(got.astype(np.float64) - exp) <= bound(x, w, b, S, pad, K, C)).all()


@pytest.mark.parametrize("offset,total", [(8, 160), (3, 135)])     # 16-byte stores or TMA boxes, 4-byte stores
@pytest.mark.parametrize("N,M,K", [(12, 128, 3), (40, 128, 1), (40, 62, 1)])
def test_tensor_core_kernel_writes_its_slice_only(N, M, K, offset, total):
    x, w, b = synth.conv_layer_case(8, N, 128, M, 29, K)
    exp = ref.conv2d(x, w, b, S=1, pad=K // 2, relu=True)
    got = G.gpu_conv(x, w, b, 1, K // 2, True, F32, c_offset=offset, c_total=total, fill=-7.0, kernel="conv_f32_tc ")
    assert (np.abs(got[:, offset:offset + M].astype(np.float64) - exp) <= bound(x, w, b, 1, K // 2, K, 128)).all()
    assert (got[:, :offset] == -7.0).all() and (got[:, offset + M:] == -7.0).all()


@pytest.mark.parametrize("K", [1, 3])
def test_exact_sums_stay_exact_and_infinities_come_through(K):
    """One kernel element per output layer: the outputs are input values, to the last bit; and an infinity, a NaN and the
    largest float end up where multiply-adds put them."""
    rng = np.random.default_rng(5)
    N, C, H = 16, 160, 27
    x = rng.standard_normal((N, C, H, H)).astype(np.float32)
    w = np.zeros((C, C, K, K), np.float32)
    w[np.arange(C), rng.permutation(C), K // 2, K // 2] = 1.0
    b = np.zeros(C, np.float32)
    exp = ref.conv2d(x, w, b, S=1, pad=K // 2, relu=False)
    np.testing.assert_array_equal(G.gpu_conv(x, w, b, 1, K // 2, False, F32, kernel="conv_f32_tc "), exp)
    x[1, 5, 3, 4], x[2, 7, 20, 20], x[3, 9, 0, 0] = np.inf, np.nan, np.finfo(np.float32).max
    with np.errstate(invalid="ignore"):
        exp = ref.conv2d(x, w, b, S=1, pad=K // 2, relu=False)
    np.testing.assert_array_equal(G.gpu_conv(x, w, b, 1, K // 2, False, F32, kernel="conv_f32_tc "), exp)


@pytest.mark.parametrize("relu", [True, False])
def test_a_bias_that_is_not_finite(relu):
    """The sum is finite, the bias is not: NaN stays NaN without ReLU and becomes 0 with it, as max(0, .) has it everywhere."""
    x, w, b = synth.conv_layer_case(6, 32, 64, 128, 27, 1)
    b[[7, 40, 100]] = np.nan, np.inf, -np.inf
    exp = ref.conv2d(x, w, np.where(np.isfinite(b), b, 0).astype(np.float32), S=1, pad=0, relu=relu)
    got = G.gpu_conv(x, w, b, 1, 0, relu, F32, kernel="conv_f32_tc ")
    special = {7: 0.0 if relu else np.nan, 40: np.inf, 100: 0.0 if relu else -np.inf}
    for m, v in special.items():
        np.testing.assert_array_equal(got[:, m], np.full_like(got[:, m], v))
    rest = np.isfinite(b)
    assert (np.abs(got.astype(np.float64) - exp) <= bound(x, w, np.nan_to_num(b, posinf=0, neginf=0), 1, 0, 1, 64))[:, rest].all()


@pytest.mark.parametrize("ex,ew", [(-139, 120), (-130, 120), (120, -130), (124, -135), (-100, -20), (75, -60), (-60, 75), (113, -100), (60, 40)])
@pytest.mark.parametrize("K", [1, 3])
def test_operands_of_any_magnitude_keep_their_bits(K, ex, ew):
    """Multiples of 2^-10 and 2^-14 times powers of two, subnormal numbers and ones that the scaled split cannot hold among
    them: the outputs are those of the unscaled operands times the same power, within the same bound."""
    x, w, b = synth.conv_layer_case(9, 20, 64, 128, 27, K)
    x, w = np.round(x * 2 ** 10) / np.float32(2 ** 10), np.round(w * 2 ** 14) / np.float32(2 ** 14)
    b[:] = 0
    x[:, 3] *= -1
    exp = ref.conv2d(x, w, b, S=1, pad=K // 2, relu=False)
    xs, ws = np.ldexp(x, ex), np.ldexp(w, ew)
    assert (np.ldexp(xs.astype(np.float64), -ex) == x).all() and (np.ldexp(ws.astype(np.float64), -ew) == w).all()
    got = np.ldexp(G.gpu_conv(xs, ws, b, 1, K // 2, False, F32, kernel="conv_f32_tc ").astype(np.float64), -ex - ew)
    # (the last term: half a unit of the smallest fp32 output)
    assert (np.abs(got - exp) <= bound(x, w, b, 1, K // 2, K, 64) + 2.0 ** (-150 - ex - ew)).all()


# (N, Cin, Cout, H, K, S, pad): a 1x1 layer with and without TMA stores, a patch, staged windows
@pytest.mark.parametrize("shape", [(30, 300, 96, 27, 1, 1, 0), (30, 300, 70, 27, 1, 1, 0), (16, 130 * 2, 100, 20, 3, 1, 1),
                                   (16, 64, 128, 56, 3, 2, 1)], ids=lambda s: "x".join(map(str, s)))
def test_sums_that_are_not_finite(shape):
    """Infinities and NaN in pixels and kernels, single ones and whole rows of them: outputs that they reach are those of
    multiply-adds, all others stay within the bound; and one infinity per image costs a few times the finite layer (up to 12
    measured), not a hundred times: only the outputs that it reaches are computed again."""
    import torch
    N, C, M, H, K, S, pad = shape
    rng = np.random.default_rng(sum(shape))
    x = rng.standard_normal((N, C, H, H)).astype(np.float32)
    w, b = synth.draw_conv_params(rng, C, M, K)

    def time_of(x):
        xd, wd, bd = G.dev_act(x, F32), G.dev_w(w, F32), G.dev_b(b)
        OH = (H + 2 * pad - K) // S + 1
        out = B.empty_device((N, OH, OH, M), F32)
        ev = [torch.cuda.Event(enable_timing=True) for _ in range(2)]
        for i in range(6):
            if i == 1:
                ev[0].record()
            B.conv_forward_ex(xd, wd, bd, out, C, M, H, H, K, S, pad, N, dtype=F32)
        ev[1].record()
        torch.cuda.synchronize()
        return ev[0].elapsed_time(ev[1])

    finite = time_of(x)
    x[:, C // 2, H // 2, H // 2] = np.inf
    assert time_of(x) < 40 * finite
    x[0, 1, :, 3], x[1, :, 2, 2], x[2, 0, 5, :], x[3] = -np.inf, np.nan, np.float32(3e38), np.inf
    # (the middle of the window: a padding zero times an infinity, which the oracle leaves out, does not occur)
    w[M - 1, 3, K // 2, K // 2], w[5, C - 1, K // 2, K // 2] = np.inf, np.nan
    with np.errstate(invalid="ignore", over="ignore"):
        exp = ref.conv2d(x, w, b, S=S, pad=pad, relu=False)
        got = G.gpu_conv(x, w, b, S, pad, False, F32, kernel="conv_f32_tc ")
        # (3e38 times a kernel value: a sum that overflows or not by the order of its terms is left out)
        unsure = np.isinf(ref.conv2d(np.abs(np.nan_to_num(x, nan=0, posinf=0, neginf=0)), np.abs(np.nan_to_num(w, nan=0, posinf=0)), np.abs(b),
                                     S=S, pad=pad, relu=False))
    fin = np.isfinite(exp)
    np.testing.assert_array_equal(got[~fin & ~unsure], exp[~fin & ~unsure])
    xf, wf = np.nan_to_num(x, nan=0, posinf=0, neginf=0), np.nan_to_num(w, nan=0, posinf=0)
    ok = fin & ~unsure
    # (outputs computed again are chains of K*K*C/32 multiply-adds and a tree of five: covered by the bound)
    assert (np.abs(got[ok].astype(np.float64) - exp[ok]) <= bound(xf, wf, b, S, pad, K, C)[ok]).all()
