"""Tensor-core tiles of 128 and 64 output layers where there are few pixels, at the edges of the rule and with ragged last
tiles, against the oracle.

Bound per output: exact products added to an fp32 accumulator that cuts sums off at 24 bits (2^-23 of what it holds) in
K*K*Cin + 2 steps, on sums no larger than the sum of |kernel * input| and |bias|, the bias as two 16-bit numbers (2^-16 of
it), the oracle's own roundings (2^-24 each); then one rounding to the 16-bit type."""
import numpy as np
import pytest

from oracle import ref
from paper_1611_07151_b200 import binding as B
from paper_1611_07151_b200 import synth
import gpu_util as G

pytestmark = pytest.mark.gpu
ULP = {B.SQN_BF16: 2.0 ** -8, B.SQN_F16: 2.0 ** -11}

# (N, Cin, Cout, H, W, K, pad)
SHAPES = [
    (17, 256, 256, 14, 14, 3, 1),       # 27 tiles of pixels: 64 layers each
    (33, 256, 256, 14, 14, 3, 1),       # 51: 128 layers
    (64, 256, 256, 14, 14, 3, 1),       # 98: as wide as they come
    (17, 512, 264, 7, 9, 1, 0),         # a last tile of 8 layers
    (20, 640, 144, 11, 11, 3, 0),       # a last tile of 16
    (21, 1024, 96, 14, 13, 1, 0),       # 64 and 32
    (60, 2048, 512, 7, 7, 1, 0),
]


@pytest.mark.parametrize("shape", SHAPES, ids=lambda s: "x".join(map(str, s)))
@pytest.mark.parametrize("dtype", [B.SQN_BF16, B.SQN_F16], ids=["bf16", "f16"])
def test_few_pixels(shape, dtype):
    import torch
    N, C, M, H, W, K, pad = shape
    rng = np.random.default_rng(sum(shape))
    tt = torch.float16 if dtype == B.SQN_F16 else torch.bfloat16
    rounded = lambda a: torch.from_numpy(np.ascontiguousarray(a, dtype=np.float32)).to(tt).float().numpy()
    x = rounded(rng.standard_normal((N, C, H, W)))
    w, b = synth.draw_conv_params(rng, C, M, K)
    w = rounded(w)
    got = G.gpu_conv(x, w, b, 1, pad, True, dtype, c_offset=8, c_total=M + 16, fill=-7.0).astype(np.float64)
    assert (got[:, :8] == -7.0).all() and (got[:, M + 8:] == -7.0).all()
    ends = [0, N - 1]
    exp = ref.conv2d(x[ends], w, b, S=1, pad=pad, relu=True).astype(np.float64)
    terms = ref.conv2d(np.abs(x[ends]), np.abs(w), np.abs(b), S=1, pad=pad, relu=False).astype(np.float64)
    n = K * K * C + 2
    err = n * (2.0 ** -23 + 2.0 ** -24) * terms + 2.0 ** -16 * np.abs(b)[None, :, None, None]
    assert (np.abs(got[ends][:, 8:M + 8] - exp) <= err + ULP[dtype] * (np.abs(exp) + err) + 2.0 ** -25).all()
    assert not np.isnan(got).any()
