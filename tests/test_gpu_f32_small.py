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

# (N, Cin, Cout, H, K, S, pad)
SHAPES = [
    (1, 512, 64, 13, 1, 1, 0),      # 12 tiles: half tiles, 32 chunks
    (1, 64, 32, 40, 3, 1, 1),       # 47 tiles
    (1, 48, 192, 27, 3, 1, 1),      # 138 tiles: three slots per warp, chunks not a multiple of 8
    (1, 64, 256, 27, 3, 1, 1),      # 184 tiles: two slots
    (1, 20, 128, 55, 3, 1, 1),      # more tiles: four warps, last chunk of 4
    (1, 16, 64, 55, 1, 1, 0),       # one chunk
    (1, 96, 16, 55, 1, 1, 0),       # narrow tiles
    (1, 40, 15, 30, 2, 1, 1),       # narrow, ragged layers, even kernel
    (2, 12, 33, 17, 3, 2, 1),       # a layer past a tile, stride
    (1, 7, 34, 19, 5, 3, 2),        # 4-byte pieces
    (1, 3, 9, 21, 7, 2, 0),         # ... narrow
    (1, 4, 4, 1, 1, 1, 0),          # one pixel
    (1, 8, 20, 3, 3, 1, 3),         # padding larger than the window
]


def check(got, x, w, b, S, pad, relu):
    exp = ref.conv2d(x, w, b, S=S, pad=pad, relu=relu)
    terms = ref.conv2d(np.abs(x), np.abs(w), np.abs(b), S=S, pad=pad, relu=False).astype(np.float64)
    assert got.shape == exp.shape
    n = w.shape[1] * w.shape[2] ** 2 + 9
    assert (np.abs(got.astype(np.float64) - exp) <= n * 2.0 ** -24 * terms).all()


@pytest.mark.parametrize("shape", SHAPES, ids=lambda s: "x".join(map(str, s)))
@pytest.mark.parametrize("relu", [True, False])
def test_small_layers_within_rounding(shape, relu):
    N, C, M, H, K, S, pad = shape
    rng = np.random.default_rng(sum(shape))
    x = rng.standard_normal((N, C, H, H + 1)).astype(np.float32)
    w, b = synth.draw_conv_params(rng, C, M, K)
    check(G.gpu_conv(x, w, b, S, pad, relu, F32), x, w, b, S, pad, relu)


@pytest.mark.parametrize("cin,s,e1,e3,h", [(96, 16, 64, 64, 55), (128, 32, 128, 128, 55), (512, 64, 256, 256, 13),
                                           (20, 12, 16, 9, 11), (10, 6, 5, 40, 9)])
def test_both_expands_of_a_fire_layer(cin, s, e1, e3, h):
    rng = np.random.default_rng(cin + s)
    x = np.abs(rng.standard_normal((1, cin, h, h + 2))).astype(np.float32)
    sq, x1, x3 = (synth.draw_conv_params(rng, *a) for a in ((cin, s, 1), (s, e1, 1), (s, e3, 3)))
    scratch = B.empty_device((1, h, h + 2, s), F32)
    out = B.empty_device((1, h, h + 2, e1 + e3), F32)
    out.fill_(float("nan"))
    B.fire_forward(G.dev_act(x, F32), G.dev_w(sq[0], F32), G.dev_b(sq[1]), G.dev_w(x1[0], F32), G.dev_b(x1[1]),
                   G.dev_w(x3[0], F32), G.dev_b(x3[1]), scratch, out, cin, s, e1, e3, h, h + 2, 1, F32)
    assert B.sqn_check() == B.SQN_OK
    squeezed = G.host_act(scratch, F32)
    check(squeezed, x, *sq, 1, 0, True)
    got = G.host_act(out, F32)
    check(got[:, :e1], squeezed, *x1, 1, 0, True)
    check(got[:, e1:], squeezed, *x3, 1, 1, True)
