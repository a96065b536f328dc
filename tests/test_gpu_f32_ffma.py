"""The exact path's FFMA kernel against the oracle, once per tile shape and kind of load (16-byte pieces, or 4-byte ones through the
table of offsets) at ragged sizes; and a reduction that the table does not hold, which only layers too large for the offsets of the
other kernels bring here.  Bar: max|delta| / max|ref| <= 1e-4, and the bound of a chain of K*K*Cin multiply-adds per output."""
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
    ((14, 4, 118, 62, 1, 2, 0), "128x128 vec"),
    ((203, 14, 1394, 2, 1, 1, 0), "128x128"),
    ((17, 4, 373, 16, 1, 1, 0), "128x96 vec"),
    ((6, 2, 92, 47, 1, 1, 0), "128x96"),
    ((40, 8, 64, 40, 2, 2, 0), "128x64 vec"),
    ((18, 3, 216, 30, 1, 2, 0), "128x64"),
    ((9, 4, 35, 77, 1, 2, 0), "128x48 vec"),
    ((9, 9, 40, 41, 3, 1, 1), "128x48"),
    ((6, 12, 28, 59, 1, 1, 0), "256x32 vec"),
    ((28, 3, 19, 40, 1, 1, 0), "256x32"),
    ((71, 96, 16, 55, 1, 1, 0), "256x16 vec"),
    ((16, 3, 13, 26, 1, 1, 0), "256x16"),
    ((1, 4, 12800, 7, 1, 1, 0), "64x128 vec"),
    ((1, 3, 12800, 7, 1, 1, 0), "64x128"),
    ((2, 12, 61, 51, 1, 1, 0), "64x64 vec"),
    ((16, 3, 38, 36, 1, 2, 0), "64x64"),
    ((1, 12, 33, 10, 1, 1, 0), "64x32 vec"),
]


@pytest.mark.parametrize("shape,variant", SHAPES, ids=["x".join(map(str, s)) for s, _ in SHAPES])
@pytest.mark.parametrize("relu", [True, False])
def test_tile_shapes(shape, variant, relu):
    N, C, M, H, K, S, pad = shape
    rng = np.random.default_rng(sum(shape))
    x = rng.standard_normal((N, C, H, H + 1)).astype(np.float32)
    w, b = synth.draw_conv_params(rng, C, M, K)
    exp = ref.conv2d(x, w, b, S=S, pad=pad, relu=relu)
    terms = ref.conv2d(np.abs(x), np.abs(w), np.abs(b), S=S, pad=pad, relu=False).astype(np.float64)
    got = G.gpu_conv(x, w, b, S, pad, relu, F32, kernel="conv_f32 " + variant)
    assert got.shape == exp.shape and G.rel_err(got, exp) <= G.TOL[F32]
    assert (np.abs(got.astype(np.float64) - exp) <= 2 * (K * K * C + 1) * 2.0 ** -24 * terms).all()       # (the oracle's roundings too)


def test_reduction_longer_than_the_table():
    """One layer of 33000 x 33000 pixels (4.4 GB), 47 x 47 windows 3000 pixels apart: beyond the 32-bit offsets of the kernel for small
    layers and the windows of the one on the tensor cores."""
    import torch
    H, K, S, M = 33000, 47, 3000, 5
    gen = torch.Generator(device="cuda").manual_seed(3)
    x = torch.randn((1, H, H, 1), generator=gen, device="cuda")
    w = torch.randn((M, K, K, 1), generator=gen, device="cuda") / K
    b = torch.randn((M,), generator=gen, device="cuda")
    n = (H - K) // S + 1
    out = torch.full((1, n, n, M), float("nan"), device="cuda")
    with G.traced() as names:
        B.conv_forward_ex(x, w, b, out, 1, M, H, H, K, S, 0, 1, dtype=F32, relu=False)
    assert B.sqn_check() == B.SQN_OK
    assert len(names) == 1 and names[0].startswith("conv_f32 ") and names[0].endswith(" no table"), names
    win = torch.stack([x[0, S * i:S * i + K, S * j:S * j + K, 0] for i in range(n) for j in range(n)]).double().reshape(n * n, K * K)
    exp = win @ w.double().reshape(M, K * K).T + b.double()
    terms = win.abs() @ w.double().abs().reshape(M, K * K).T + b.double().abs()
    assert ((out.double().reshape(n * n, M) - exp).abs() <= (K * K + 1) * 2.0 ** -24 * terms).all()
