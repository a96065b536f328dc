"""The pooled kernel's tile sizes (256, 144 and 128 pixels) on both sides of the lines between them: one convolution with its
max-pool, against the unfused pair of calls bit for bit, and against the oracle at both ends of the batch (16-bit operands
and output: 2e-2 of the largest value, as the other pooled cases)."""
import numpy as np
import pytest

from oracle import ref
from paper_1611_07151_b200 import binding as B
from paper_1611_07151_b200 import synth
import gpu_util as G

pytestmark = pytest.mark.gpu

# (N, Cin, Cout, H, W, K, S, pad)
CASES = [
    (18, 3, 96, 227, 227, 7, 2, 0),     # 128 pixels: 144 strips
    (19, 3, 96, 227, 227, 7, 2, 0),     # 144 pixels: 133 strips
    (22, 3, 96, 227, 227, 7, 2, 0),     # 256 pixels
    (40, 3, 32, 111, 99, 7, 2, 0),      # ... ragged, other layer counts
    (50, 16, 64, 35, 41, 3, 1, 1),      # 144 or 128 pixels, several strips per CTA
    (37, 32, 128, 39, 40, 3, 1, 1),
    (75, 32, 96, 36, 36, 1, 1, 0),
]


@pytest.mark.parametrize("case", CASES, ids=lambda c: "x".join(map(str, c)))
@pytest.mark.parametrize("dtype", [B.SQN_BF16, B.SQN_F16], ids=["bf16", "f16"])
def test_pooled_layer(case, dtype):
    N, C, M, H, W, K, S, pad = case
    rng = np.random.default_rng(sum(case))
    x = synth.draw_input(rng, (N, C, H, W))
    w, b = synth.draw_conv_params(rng, C, M, K)
    got = G.gpu_conv(x, w, b, S, pad, True, dtype, fuse_maxpool=True)
    full = G.gpu_conv(x, w, b, S, pad, True, dtype)
    np.testing.assert_array_equal(got, ref.maxpool(full, 3, 2))
    ends = [0, N - 1]
    exp = ref.maxpool(ref.conv2d(x[ends], w, b, S=S, pad=pad, relu=True), 3, 2)
    assert G.rel_err(got[ends], exp) <= 2e-2
