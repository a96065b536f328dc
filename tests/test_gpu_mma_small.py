"""The 16-bit kernel for small layers (the reduction split over the warps of a CTA) against the oracle, at the edges of its tiles,
chunks of 32 and launch shapes: single layers of more than 128 output layers, fire layers too wide for the one-kernel path, and
the fire layers of the network at a batch of 1.

Bound per output: the products are exact, each is added to an fp32 sum that the matrix units may cut to 24 bits (2^-23 of
what it holds), and so are at most 8 partial sums and the bias: K*K*Cin + 9 steps on sums no larger than the sum of
|kernel * input| and |bias|; then one rounding to the 16-bit type."""
import numpy as np
import pytest

from oracle import ref
from paper_1611_07151_b200 import binding as B
from paper_1611_07151_b200 import synth
import gpu_util as G

pytestmark = pytest.mark.gpu
ULP = {B.SQN_BF16: 2.0 ** -8, B.SQN_F16: 2.0 ** -11}

# (N, Cin, Cout, H, W, K, pad), the variant that runs
SHAPES = [
    ((1, 32, 264, 9, 7, 1, 0), "1 warps, 2 slots"),         # one chunk, layers past a tile
    ((1, 48, 144, 12, 8, 1, 0), "2 warps, 2 slots"),        # two chunks, the last of 16
    ((1, 112, 160, 5, 13, 1, 0), "4 warps, 2 slots"),       # four chunks
    ((1, 512, 1000, 13, 13, 1, 0), "8 warps, 2 slots"),     # 192 tiles, 8 pixels past a tile, 8 layers past a tile
    ((1, 512, 512, 7, 7, 3, 1), "8 warps, 3 slots"),        # 144 chunks
    ((1, 16, 48, 1, 1, 3, 1), "8 warps, 3 slots"),          # one pixel
    ((1, 176, 256, 3, 10, 5, 2), "8 warps, 3 slots"),
    ((1, 64, 256, 13, 13, 3, 0), "8 warps, 3 slots"),
]

def check(got, x, w, b, pad, relu, dtype):
    exp = ref.conv2d(x, w, b, S=1, pad=pad, relu=relu).astype(np.float64)
    terms = ref.conv2d(np.abs(x), np.abs(w), np.abs(b), S=1, pad=pad, relu=False).astype(np.float64)
    assert got.shape == exp.shape
    n = w.shape[1] * w.shape[2] ** 2 + 9
    err = n * 2.0 ** -23 * terms + n * 2.0 ** -24 * terms          # the kernel's sums, the fp32 oracle's
    assert (np.abs(got.astype(np.float64) - exp) <= err + ULP[dtype] * (np.abs(exp) + err) + 2.0 ** -25).all()


def rounded(a, dtype):
    import torch
    t = torch.from_numpy(np.ascontiguousarray(a, dtype=np.float32))
    return (t.half() if dtype == B.SQN_F16 else t.bfloat16()).float().numpy()


@pytest.mark.parametrize("shape,variant", SHAPES, ids=["x".join(map(str, s)) for s, _ in SHAPES])
@pytest.mark.parametrize("dtype", [B.SQN_BF16, B.SQN_F16], ids=["bf16", "f16"])
def test_single_layers(shape, variant, dtype):
    N, C, M, H, W, K, pad = shape
    rng = np.random.default_rng(sum(shape))
    x = rounded(rng.standard_normal((N, C, H, W)), dtype)
    w, b = synth.draw_conv_params(rng, C, M, K)
    w = rounded(w, dtype)
    for relu in (True, False):
        check(G.gpu_conv(x, w, b, 1, pad, relu, dtype, kernel="conv_mma_small, " + variant), x, w, b, pad, relu, dtype)


@pytest.mark.parametrize("cin,s,e1,e3,h,batch,variant", [
    (512, 64, 256, 256, 13, 1, "8 warps, 3 slots"),
    (512, 64, 256, 256, 13, 2, "8 warps, 2 slots"),         # 208 tiles of both expands
    (512, 64, 256, 256, 13, 4, "4 warps, 3 slots"),         # 400
    (512, 64, 256, 256, 13, 6, "4 warps, 2 slots"),         # 592
    (384, 48, 192, 192, 27, 1, "4 warps, 3 slots"),
    (64, 80, 32, 48, 6, 1, "8 warps, 3 slots")])
@pytest.mark.parametrize("dtype", [B.SQN_BF16, B.SQN_F16], ids=["bf16", "f16"])
def test_fire_layers(cin, s, e1, e3, h, batch, variant, dtype):
    rng = np.random.default_rng(cin + s)
    x = rounded(np.abs(rng.standard_normal((batch, cin, h, h + 2))), dtype)
    sq, x1, x3 = ((rounded(w, dtype), b) for w, b in
                  (synth.draw_conv_params(rng, *a) for a in ((cin, s, 1), (s, e1, 1), (s, e3, 3))))
    scratch = B.empty_device((batch, h, h + 2, s), dtype)
    out = B.empty_device((batch, h, h + 2, e1 + e3), dtype)
    out.fill_(float("nan"))
    args = (G.dev_act(x, dtype), G.dev_w(sq[0], dtype), G.dev_b(sq[1]), G.dev_w(x1[0], dtype), G.dev_b(x1[1]), G.dev_w(x3[0], dtype),
            G.dev_b(x3[1]), scratch, out, cin, s, e1, e3, h, h + 2, batch, dtype)
    with G.traced() as names:
        B.fire_forward(*args)
    assert len(names) == 2 and names[0].startswith("conv_mma_small, ") and names[1] == "conv_mma_small x 2, " + variant, names
    assert B.sqn_check() == B.SQN_OK
    squeezed = G.host_act(scratch, dtype)
    check(squeezed, x, *sq, 0, True, dtype)
    got = G.host_act(out, dtype)
    check(got[:, :e1], squeezed, *x1, 0, True, dtype)
    check(got[:, e1:], squeezed, *x3, 1, True, dtype)


@pytest.mark.parametrize("dtype", [B.SQN_BF16, B.SQN_F16], ids=["bf16", "f16"])
def test_net_of_one_image_layer_by_layer(dtype):
    """Every stored map against the oracle's layer on the stored map before it: the rounding of the squeeze map within (up to
    one unit, taken through the expands' kernels) is the only error besides a layer's own."""
    import torch
    names = [n for n, *_ in synth.SQUEEZENET_CONVS]
    x, params = synth.squeezenet_case(5, 1)
    ws = [G.dev_w(params[n][0], dtype) for n in names]
    bs = [G.dev_b(params[n][1]) for n in names]
    net = B.squeezenet_create(ws, bs, dtype, 1)
    work = torch.empty(B.squeezenet_workspace_bytes(net, 1), dtype=torch.uint8, device="cuda")
    logits = torch.empty((1, 1000), device="cuda")
    B.squeezenet_forward(net, G.dev_act(x, dtype), logits, None, work, 1)
    assert B.sqn_check() == B.SQN_OK

    def stored(name):
        ptr, C, H, W = B.squeezenet_layer_output(net, name, work, 1)
        off = (ptr - work.data_ptr()) // 2
        el = work.view(torch.float16 if dtype == B.SQN_F16 else torch.bfloat16)[off:off + C * H * W]
        return np.ascontiguousarray(el.view(H, W, C).permute(2, 0, 1)[None].float().cpu().numpy())

    prev = "pool1"
    for i in range(2, 10):
        name = "fire%d" % i
        w = {k: rounded(params["%s_%s" % (name, k)][0], dtype) for k in ("sq", "e1", "e3")}
        b = {k: params["%s_%s" % (name, k)][1] for k in ("sq", "e1", "e3")}
        s = rounded(ref.conv2d(stored(prev), w["sq"], b["sq"], S=1, pad=0, relu=True), dtype)
        got, e = stored(name), w["e1"].shape[0]
        for k, part, pad in (("e1", got[:, :e], 0), ("e3", got[:, e:], 1)):
            exp = ref.conv2d(s, w[k], b[k], S=1, pad=pad, relu=True).astype(np.float64)
            slack = ref.conv2d(np.abs(s), np.abs(w[k]), np.abs(b[k]), S=1, pad=pad, relu=False).astype(np.float64)
            n = w[k].shape[1] * w[k].shape[2] ** 2 + 9
            err = (2 * ULP[dtype] + n * 2.0 ** -22) * slack
            assert (np.abs(part - exp) <= err + ULP[dtype] * (np.abs(exp) + err)).all(), (name, k)
        prev = "pool%d" % i if i in (4, 8) else name
    B.squeezenet_destroy(net)
