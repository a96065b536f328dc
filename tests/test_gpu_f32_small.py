"""The exact path's kernel for small layers (the reduction split over the warps of a CTA) against the oracle, at the edges of
its tiles, chunks of 16 and launch shapes, and two layers in one launch through fire_forward.

Bound per output: each warp's partial sum is a chain of multiply-adds, the partial sums and the bias are added after it, one
rounding (2^-24) each: at most K*K*Cin + 9 of them on sums no larger than the sum of |kernel * input| and |bias|."""
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
    ((1, 512, 64, 13, 1, 1, 0), "16x32 vec, 8 warps, 3 slots"),     # 12 tiles: half tiles, 32 chunks
    ((1, 64, 32, 40, 3, 1, 1), "16x32 vec, 8 warps, 3 slots"),
    ((1, 48, 192, 27, 3, 1, 1), "32x32 vec, 8 warps, 3 slots"),     # 144 tiles, chunks not a multiple of 8
    ((1, 64, 256, 27, 3, 1, 1), "32x32 vec, 8 warps, 2 slots"),     # 192 tiles
    ((1, 20, 128, 55, 3, 1, 1), "32x32 vec, 4 warps, 3 slots"),     # more tiles, last chunk of 4
    ((1, 16, 64, 56, 1, 3, 0), "16x32 vec, 4 warps, 3 slots"),      # one chunk
    ((1, 96, 16, 55, 1, 1, 0), "32x16 vec, 8 warps, 3 slots"),      # narrow tiles
    ((1, 40, 15, 30, 2, 1, 1), "32x16 vec, 8 warps, 3 slots"),      # ... ragged layers, even kernel
    ((3, 64, 13, 44, 3, 1, 1), "64x16 vec, 8 warps, 3 slots"),
    ((5, 64, 13, 55, 3, 1, 1), "64x16 vec, 8 warps, 2 slots"),
    ((31, 4, 1, 29, 1, 2, 0), "64x16 vec, 4 warps, 3 slots"),       # one output layer
    ((2, 12, 33, 17, 3, 2, 1), "16x32 vec, 8 warps, 3 slots"),      # a layer past a tile, stride
    ((8, 64, 128, 33, 3, 2, 1), "32x32 vec, 8 warps, 2 slots"),
    ((1, 7, 34, 19, 5, 3, 2), "16x32, 8 warps, 3 slots"),           # 4-byte pieces
    ((4, 35, 72, 45, 3, 2, 1), "32x32, 8 warps, 2 slots"),
    ((12, 130, 128, 28, 1, 2, 0), "32x32, 4 warps, 3 slots"),       # ... windows apart from one another
    ((1, 3, 9, 21, 7, 2, 0), "32x16, 8 warps, 3 slots"),            # ... narrow
    ((46, 5, 1, 13, 3, 1, 1), "64x16, 8 warps, 3 slots"),
    ((6, 21, 11, 55, 3, 1, 1), "64x16, 8 warps, 2 slots"),
    ((20, 5, 9, 44, 3, 1, 1), "64x16, 4 warps, 3 slots"),
    ((1, 40, 20, 3, 1, 4, 0), "16x32 vec, 8 warps, 3 slots"),       # one pixel
    ((1, 8, 20, 3, 3, 1, 3), "16x32 vec, 8 warps, 3 slots"),        # padding larger than the window
]

def check(got, x, w, b, S, pad, relu):
    exp = ref.conv2d(x, w, b, S=S, pad=pad, relu=relu)
    terms = ref.conv2d(np.abs(x), np.abs(w), np.abs(b), S=S, pad=pad, relu=False).astype(np.float64)
    assert got.shape == exp.shape
    n = w.shape[1] * w.shape[2] ** 2 + 9
    assert (np.abs(got.astype(np.float64) - exp) <= n * 2.0 ** -24 * terms).all()


@pytest.mark.parametrize("shape,variant", SHAPES, ids=["x".join(map(str, s)) for s, _ in SHAPES])
@pytest.mark.parametrize("relu", [True, False])
def test_small_layers_within_rounding(shape, variant, relu):
    N, C, M, H, K, S, pad = shape
    rng = np.random.default_rng(sum(shape))
    x = rng.standard_normal((N, C, H, H + 1)).astype(np.float32)
    w, b = synth.draw_conv_params(rng, C, M, K)
    check(G.gpu_conv(x, w, b, S, pad, relu, F32, kernel="conv_f32_small " + variant), x, w, b, S, pad, relu)


@pytest.mark.parametrize("cin,s,e1,e3,h", [(96, 16, 64, 64, 55), (128, 32, 128, 128, 55), (512, 64, 256, 256, 13),
                                           (20, 12, 16, 9, 11), (10, 6, 5, 40, 9)])
def test_both_expands_of_a_fire_layer(cin, s, e1, e3, h):
    rng = np.random.default_rng(cin + s)
    x = np.abs(rng.standard_normal((1, cin, h, h + 2))).astype(np.float32)
    sq, x1, x3 = (synth.draw_conv_params(rng, *a) for a in ((cin, s, 1), (s, e1, 1), (s, e3, 3)))
    scratch = B.empty_device((1, h, h + 2, s), F32)
    out = B.empty_device((1, h, h + 2, e1 + e3), F32)
    out.fill_(float("nan"))
    args = (G.dev_act(x, F32), G.dev_w(sq[0], F32), G.dev_b(sq[1]), G.dev_w(x1[0], F32), G.dev_b(x1[1]), G.dev_w(x3[0], F32),
            G.dev_b(x3[1]), scratch, out, cin, s, e1, e3, h, h + 2, 1, F32)
    with G.traced() as names:
        B.fire_forward(*args)
    assert B.sqn_check() == B.SQN_OK
    assert len(names) == 2 and names[1].startswith("conv_f32_small x 2 "), names
    squeezed = G.host_act(scratch, F32)
    check(squeezed, x, *sq, 1, 0, True)
    got = G.host_act(out, F32)
    check(got[:, :e1], squeezed, *x1, 1, 0, True)
    check(got[:, e1:], squeezed, *x3, 1, 1, True)
