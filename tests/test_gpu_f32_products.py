"""The fp32 kernels of small layers on the matrix instructions (three bf16 numbers per operand): operands of any magnitude, sums
that are not finite, and the stem with its max-pool in one launch, against the oracle.

Bound per output, S = the sum of |kernel * input| over the window: the products left out are below 2^-22 of the operands'
product, K*K*Cin + 9 additions of at most 2^-23 of what they hold."""
import numpy as np
import pytest

from oracle import ref
from paper_1611_07151_b200 import binding as B
from paper_1611_07151_b200 import synth
import gpu_util as G

pytestmark = pytest.mark.gpu
F32 = B.SQN_F32


def bound(x, w, b, S, pad):
    terms = ref.conv2d(np.abs(x), np.abs(w), np.abs(b), S=S, pad=pad, relu=False).astype(np.float64)
    return (2.0 ** -22 + (w.shape[1] * w.shape[2] ** 2 + 9) * 2.0 ** -23) * terms


@pytest.mark.parametrize("ex,ew", [(-139, 120), (120, -130), (-100, -20), (75, -60), (113, -100), (60, 40)])
def test_operands_of_any_magnitude(ex, ew):
    """Multiples of 2^-10 and 2^-14 times powers of two: the outputs are those of the unscaled operands times the same power."""
    x, w, b = synth.conv_layer_case(9, 1, 64, 256, 27, 3)
    x, w = np.round(x * 2 ** 10) / np.float32(2 ** 10), np.round(w * 2 ** 14) / np.float32(2 ** 14)
    b[:] = 0
    x[:, 3] *= -1
    exp = ref.conv2d(x, w, b, S=1, pad=1, relu=False)
    got = G.gpu_conv(np.ldexp(x, ex), np.ldexp(w, ew), b, 1, 1, False, F32, kernel="conv_f32_small 32x32 vec, 8 warps, 2 slots, products")
    got = np.ldexp(got.astype(np.float64), -ex - ew)
    # (the last term: half a unit of the smallest fp32 output)
    assert (np.abs(got - exp) <= bound(x, w, b, 1, 1) + 2.0 ** (-150 - ex - ew)).all()


# (N, Cin, Cout, H, K, S, pad), the variant that runs
VARIANTS = [((1, 64, 256, 27, 3, 1, 1), "32x32 vec, 8 warps, 2 slots"), ((1, 128, 32, 55, 1, 1, 0), "32x32 vec, 8 warps, 3 slots"),
            ((2, 20, 33, 17, 3, 2, 1), "16x32 vec, 8 warps, 3 slots"), ((8, 64, 128, 33, 3, 2, 1), "32x32 vec, 8 warps, 2 slots"),
            ((13, 20, 36, 44, 5, 2, 2), "32x40 vec, 8 warps, 2 slots"), ((9, 12, 48, 50, 3, 2, 1), "32x48 vec, 8 warps, 2 slots"),
            ((9, 20, 36, 44, 5, 2, 2), "32x32 vec, 8 warps, 2 slots"), ((6, 12, 48, 50, 3, 2, 1), "32x32 vec, 8 warps, 2 slots"),
            ((17, 12, 96, 34, 3, 2, 1), "32x32 vec, 4 warps, 3 slots")]


@pytest.mark.parametrize("shape,variant", VARIANTS, ids=lambda s: "x".join(map(str, s)) if isinstance(s, tuple) else s)
def test_sums_finite_and_not(shape, variant):
    N, C, M, H, K, S, pad = shape
    rng = np.random.default_rng(sum(shape))
    x = rng.standard_normal((N, C, H, H)).astype(np.float32)
    w, b = synth.draw_conv_params(rng, C, M, K)
    for special in (False, True):
        if special:
            x[0, 1, :, 3], x[0, 2, 9, 9], x[N - 1, 0, 5, 5] = np.inf, np.nan, -np.inf
            w[M - 1, 3, K // 2, K // 2], w[5, C - 1, K // 2, K // 2] = np.inf, np.nan
        with np.errstate(invalid="ignore", over="ignore"):
            exp = ref.conv2d(x, w, b, S=S, pad=pad, relu=False)
        got = G.gpu_conv(x, w, b, S, pad, False, F32, kernel="conv_f32_small %s, products" % variant)
        fin = np.isfinite(exp)
        np.testing.assert_array_equal(got[~fin], exp[~fin])
        xf, wf = np.where(np.isfinite(x), x, 0), np.where(np.isfinite(w), w, 0)
        assert (np.abs(got[fin].astype(np.float64) - exp[fin]) <= bound(xf, wf, b, S, pad)[fin]).all()
        if not special:
            check_precision(got, x, w, b, S, pad)


def check_precision(got, x, w, b, S, pad):
    """Against 64 bits.  2-norm: 0.7e-7 to 1.4e-7 measured; without the least of the five correction products (2^-17 of a product, in random
    directions) it would be 1e-6.  Largest: the products left out, two cuts of 2^-23 of what a chunk of 16 holds, a rounding for every chunk, and
    twelve for corrections, the warps' partial sums and the bias, on sums no larger than the sum of |kernel * input|."""
    K = w.shape[2]
    exp = exact(x, w, pad, S) + b[None, :, None, None].astype(np.float64)
    terms = exact(np.abs(x), np.abs(w), pad, S) + np.abs(b)[None, :, None, None]
    d = got.astype(np.float64) - exp
    assert np.linalg.norm(d) <= 3e-7 * np.linalg.norm(exp), np.linalg.norm(d) / np.linalg.norm(exp)
    assert (np.abs(d) <= (2.0 ** -22 + 2 * 2.0 ** -23 + (w.shape[1] * K * K / 16 + 12) * 2.0 ** -24) * terms).all()


# (images, input, squeeze, expand layers, rows), the variant of both expands' launch
PAIRS = [((1, 128, 32, 128, 55), "32x32 vec, 4 warps, 3 slots"), ((1, 256, 32, 128, 27), "32x32 vec, 8 warps, 2 slots"),
         ((1, 256, 48, 64, 19), "16x32 vec, 8 warps, 3 slots")]


@pytest.mark.parametrize("shape,variant", PAIRS, ids=lambda s: "x".join(map(str, s)) if isinstance(s, tuple) else s)
@pytest.mark.parametrize("special", [False, True])
def test_both_expands_finite_and_not(shape, variant, special):
    N, cin, s, e, h = shape
    rng = np.random.default_rng(sum(shape))
    x = np.abs(rng.standard_normal((N, cin, h, h + 1))).astype(np.float32)
    sq, x1, x3 = (synth.draw_conv_params(rng, *a) for a in ((cin, s, 1), (s, e, 1), (s, e, 3)))
    if special:
        x1[0][5, 2, 0, 0], x3[0][e - 1, 0, 1, 1], x3[0][3, 1, 1, 1] = np.inf, np.nan, -np.inf
        x[0, 3, 4, 5] = np.inf
    scratch, out = B.empty_device((N, h, h + 1, s), F32), B.empty_device((N, h, h + 1, 2 * e), F32)
    with G.traced() as names:
        B.fire_forward(G.dev_act(x, F32), G.dev_w(sq[0], F32), G.dev_b(sq[1]), G.dev_w(x1[0], F32), G.dev_b(x1[1]), G.dev_w(x3[0], F32),
                       G.dev_b(x3[1]), scratch, out, cin, s, e, e, h, h + 1, N, F32)
    assert B.sqn_check() == B.SQN_OK
    assert len(names) == 2 and names[1] == "conv_f32_small x 2 %s, products" % variant, names
    squeezed, got = G.host_act(scratch, F32), G.host_act(out, F32)
    for part, (w, b), pad in ((got[:, :e], x1, 0), (got[:, e:], x3, 1)):
        with np.errstate(invalid="ignore", over="ignore"):
            exp = ref.conv2d(squeezed, w, b, S=1, pad=pad, relu=False)
        fin = np.isfinite(exp)
        assert special != fin.all()
        exp = np.where(np.isnan(exp), 0, np.maximum(exp, 0))            # (max(0, NaN) = 0)
        np.testing.assert_array_equal(part[~fin], exp[~fin])
        xf, wf = np.where(np.isfinite(squeezed), squeezed, 0), np.where(np.isfinite(w), w, 0)
        assert (np.abs(part[fin].astype(np.float64) - exp[fin]) <= bound(xf, wf, b, 1, pad)[fin]).all()
        if not special:
            full = exact(squeezed, w, pad) + b[None, :, None, None].astype(np.float64)
            d = part.astype(np.float64) - np.maximum(full, 0)
            assert np.linalg.norm(d) <= 3e-7 * np.linalg.norm(np.maximum(full, 0))


def relu_map(rng, shape):
    """Positive values and as many zeros, what a layer behind a ReLU reads."""
    return np.maximum(rng.standard_normal(shape), 0).astype(np.float32)


def exact(x, w, pad, S=1):
    import torch
    return torch.nn.functional.conv2d(torch.from_numpy(x).double(), torch.from_numpy(w).double(), stride=S, padding=pad).numpy()


def signed(got, exp):
    """The error of one sign: its mean towards larger magnitudes over the mean magnitude."""
    return float(((got.astype(np.float64) - exp) * np.sign(exp)).sum() / np.abs(exp).sum())


# Products of sums that the matrix instructions cut off: without what is added back 5e-9 and 6.2e-9 (kernels of both signs, of one), with
# 1e-8 added back 4.9e-9 and 3.8e-9 in the other direction; what is added back leaves less than half of either.  The mean of 46000 outputs
# and more, each off by 0.8e-7 of the mean magnitude (0.5e-7), is itself within 4e-10 of its expectation.
@pytest.mark.parametrize("signs,most", [("both", 2.5e-9), ("one", 2.7e-9)])
def test_no_error_of_one_sign_on_maps_behind_a_relu(signs, most):
    means = []
    for seed, (N, C, M, H, K, variant) in enumerate([(1, 64, 256, 27, 3, "32x32 vec, 8 warps, 2 slots"), (1, 256, 128, 40, 1, "32x32 vec, 8 warps, 2 slots"),
                                                     (2, 48, 96, 39, 3, "32x32 vec, 8 warps, 2 slots"), (4, 512, 64, 13, 1, "16x32 vec, 8 warps, 3 slots")]):
        rng = np.random.default_rng(seed)
        x = relu_map(rng, (N, C, H, H))
        w, b = synth.draw_conv_params(rng, C, M, K)
        w = np.abs(w) if signs == "one" else w
        got = G.gpu_conv(x, w, np.zeros_like(b), 1, K // 2, False, F32, kernel="conv_f32_small %s, products" % variant)
        means.append(signed(got, exact(x, w, K // 2)))
    assert abs(np.mean(means)) <= most, means


def test_a_chain_of_layers():
    """Eight 3x3 layers with ReLU, one after the other: an error of one sign would add up (8 x 5e-9 without what is added back)."""
    rng = np.random.default_rng(3)
    x = relu_map(rng, (2, 48, 39, 39))
    got, exp = x, x.astype(np.float64)
    for i in range(8):
        w, b = synth.draw_conv_params(rng, 48 if i == 0 else 96, 96, 3)
        b[:] = 0
        got = G.gpu_conv(got, w, b, 1, 1, True, F32, kernel="conv_f32_small 32x32 vec, 8 warps, 2 slots, products")
        exp = np.maximum(exact(exp, w.astype(np.float64), 1), 0)
    assert abs(signed(got, exp)) <= 8 * 2.5e-9, signed(got, exp)
    err = np.linalg.norm(got - exp) / np.linalg.norm(exp)
    assert err <= 3e-7, err                     # (each layer's own 1e-7, most of it averaged out by the next)


# (N, Cin, Cout, H, W, K, S, pad), the variant that runs; microseconds with multiply-adds / products as measured
MULTIPLY_ADDS = [((9, 64, 221, 19, 12, 1, 2, 0), "32x32 vec, 8 warps, 3 slots"),        # 2.7 / 3.3
                 ((1, 128, 128, 30, 30, 1, 1, 0), "32x32 vec, 8 warps, 3 slots"),       # 3.3 / 3.6
                 ((1, 4, 80, 53, 26, 1, 2, 0), "16x32 vec, 4 warps, 3 slots"),          # 1.9 / 2.1
                 ((5, 476, 364, 13, 15, 1, 1, 0), "32x32 vec, 4 warps, 3 slots")]       # 15.8 / 17.2


@pytest.mark.parametrize("shape,variant", MULTIPLY_ADDS, ids=lambda s: "x".join(map(str, s)) if isinstance(s, tuple) else s)
def test_multiply_adds_where_they_are_faster(shape, variant):
    N, C, M, H, W, K, S, pad = shape
    x, w, b = B.empty_device((N, H, W, C)), B.empty_device((M, K, K, C)), B.empty_device((M,))
    out = B.empty_device((N, (H + 2 * pad - K) // S + 1, (W + 2 * pad - K) // S + 1, M))
    with G.traced() as names:
        B.conv_forward_ex(x, w, b, out, C, M, H, W, K, S, pad, N)
    assert B.sqn_check() == B.SQN_OK
    assert names == ["conv_f32_small " + variant]


def stem_of_one_image(special):
    """(image, kernels, bias, the stored convolution, the stored pooled map)."""
    import torch
    x, params = synth.squeezenet_case(37, 1)
    if special:
        x[0, 1, 100, 50], x[0, 2, 226, 226], x[0, 0, 0, 30] = np.inf, np.nan, np.float32(3e38)
    names = [n for n, *_ in synth.SQUEEZENET_CONVS]
    ws, bs = [G.dev_w(params[n][0], F32) for n in names], [G.dev_b(params[n][1]) for n in names]
    net = B.squeezenet_create(ws, bs, F32, 1)
    work = torch.empty(B.squeezenet_workspace_bytes(net, 1), dtype=torch.uint8, device="cuda")
    logits = torch.empty((1, 1000), device="cuda")
    with G.traced() as launched:
        B.squeezenet_forward(net, G.dev_act(x, F32), logits, None, work, 1)
    assert B.sqn_check() == B.SQN_OK
    assert launched[0] == "stem_small_f32", launched
    maps = []
    for name in ("conv1", "pool1"):
        ptr, C, H, W = B.squeezenet_layer_output(net, name, work, 1)
        off = (ptr - work.data_ptr()) // 4
        maps.append(work.view(torch.float32)[off:off + C * H * W].view(H, W, C).permute(2, 0, 1)[None].cpu().numpy())
    B.squeezenet_destroy(net)
    return (x,) + params["conv1"] + tuple(maps)


@pytest.mark.parametrize("special", [False, True])
def test_stem_of_one_image(special):
    x, w, b, *maps = stem_of_one_image(special)
    with np.errstate(invalid="ignore", over="ignore"):
        exp = ref.conv2d(x, w, b, S=2, pad=0, relu=False)
        low = ref.conv2d(np.abs(np.where(np.isfinite(x), x, 0)), np.abs(w), np.abs(b), S=2, pad=0, relu=False)
    if not special:
        full = np.maximum(exact(x, w, 0, 2) + b[None, :, None, None].astype(np.float64), 0)
        assert np.linalg.norm(maps[0] - full) <= 3e-7 * np.linalg.norm(full)
    exp = np.where(np.isnan(exp), 0, np.maximum(exp, 0)).astype(np.float64)          # (max(0, NaN) = 0)
    fin = np.isfinite(exp) & np.isfinite(low)
    np.testing.assert_array_equal(maps[0][np.isposinf(exp) & np.isfinite(low)], np.inf)
    assert (np.abs(maps[0][fin] - exp[fin]) <= (2.0 ** -22 + 156 * 2.0 ** -23) * low[fin].astype(np.float64)).all()
    # the pooled map: the maximum of the stored one, exactly; where a tile was computed again and its neighbours, which share pixels
    # with it, were not, up to both tiles' bounds
    windows = lambda a: np.max([a[:, i:i + 109:2, j:j + 109:2] for i in range(3) for j in range(3)], axis=0)
    pooled, most = windows(maps[0][0]), windows(low[0].astype(np.float64))
    if special:
        same = pooled == maps[1][0]
        with np.errstate(invalid="ignore"):
            near = np.abs(pooled - maps[1][0]) <= 2 * (2.0 ** -22 + 156 * 2.0 ** -23) * most
        assert (same | near).all() and same.mean() > 0.99
    else:
        np.testing.assert_array_equal(maps[1][0], pooled)


def test_a_stem_with_an_infinity_pools_the_map_that_it_stores():
    """Tiles share pixels: one that is computed again must not change the pixels whose sums were finite."""
    *_, conv, pool = stem_of_one_image(True)
    windows = np.max([conv[0][:, i:i + 109:2, j:j + 109:2] for i in range(3) for j in range(3)], axis=0)
    np.testing.assert_array_equal(pool[0], windows)
