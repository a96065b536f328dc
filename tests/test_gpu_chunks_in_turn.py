"""16-bit layers whose epilogue's two groups of warps take chunks in turn, and the layers next to them that do not: the variant by
name, the values against the oracle.

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

# (N, Cin, Cout, H, W, K), layers of a tile, in turn
LAYERS = [
    ((30, 64, 256, 41, 39, 1), 256, True),          # four chunks, several tiles per CTA
    ((20, 160, 160, 52, 57, 1), 160, True),         # five: the groups change places from tile to tile
    ((33, 48, 400, 31, 28, 1), 256, True),          # a last column of tiles with fewer chunks
    ((42, 240, 240, 29, 13, 1), 240, True),         # 15 chunks of 16 layers, one tile per CTA
    ((13, 32, 96, 39, 10, 3), 96, True),            # a patch
    ((52, 288, 384, 11, 28, 1), 256, False),        # a longer reduction, several tiles per CTA
    ((28, 80, 384, 21, 12, 1), 256, False),         # a short one, one tile per CTA
    ((30, 16, 240, 56, 23, 3), 240, False),         # a patch, several tiles per CTA
]


@pytest.mark.parametrize("shape,bn,turn", LAYERS, ids=lambda s: "x".join(map(str, s)) if isinstance(s, tuple) else str(s))
@pytest.mark.parametrize("dtype", [B.SQN_BF16, B.SQN_F16], ids=["bf16", "f16"])
def test_chunks_in_turn(shape, bn, turn, dtype):
    import torch
    N, C, M, H, W, K = shape
    rng = np.random.default_rng(sum(shape))
    tt = torch.float16 if dtype == B.SQN_F16 else torch.bfloat16
    rounded = lambda a: torch.from_numpy(np.ascontiguousarray(a, dtype=np.float32)).to(tt).float().numpy()
    x = rounded(rng.standard_normal((N, C, H, W)))
    w, b = synth.draw_conv_params(rng, C, M, K)
    w = rounded(w)
    got = G.gpu_conv(x, w, b, 1, K // 2, True, dtype, c_offset=8, c_total=M + 16, fill=-7.0).astype(np.float64)
    with G.traced() as names:
        B.conv_forward_ex(G.dev_act(x, dtype), G.dev_w(w, dtype), G.dev_b(b), B.empty_device((N, H, W, M), dtype), C, M, H, W, K, 1, K // 2, N, dtype=dtype)
    name = names[0].replace(", a shorter last chunk", "")
    assert len(names) == 1 and name == "conv_tc, %d layers%s" % (bn, ", chunks in turn" if turn else ""), names
    assert (got[:, :8] == -7.0).all() and (got[:, M + 8:] == -7.0).all()
    some = [0, N // 2, N - 1]
    exp = ref.conv2d(x[some], w, b, S=1, pad=K // 2, relu=True).astype(np.float64)
    terms = ref.conv2d(np.abs(x[some]), np.abs(w), np.abs(b), S=1, pad=K // 2, relu=False).astype(np.float64)
    err = (K * K * C + 2) * (2.0 ** -23 + 2.0 ** -24) * terms + 2.0 ** -16 * np.abs(b)[None, :, None, None]
    assert (np.abs(got[some][:, 8:M + 8] - exp) <= err + ULP[dtype] * (np.abs(exp) + err) + 2.0 ** -25).all()
