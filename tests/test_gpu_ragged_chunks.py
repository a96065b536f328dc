"""Tensor-core layers without a patch whose input layers are no multiple of 64: chunks of 64 with a shorter last one, kernels
resident and streamed, flat and tap by tap, against the oracle.

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
    (40, 48, 64, 30, 31, 1, 0),         # one chunk of three MMAs
    (40, 80, 16, 33, 29, 1, 0),         # a last chunk of one MMA
    (40, 96, 128, 27, 27, 1, 0),        # ... of two
    (21, 112, 520, 14, 15, 1, 0),       # ... of three, three columns of tiles
    (4, 240, 128, 19, 18, 3, 1),        # kernels streamed
    (10, 208, 240, 10, 23, 3, 1),
    (20, 80, 256, 17, 9, 5, 2),
    (16, 144, 32, 20, 21, 3, 0),
]


@pytest.mark.parametrize("shape", SHAPES, ids=lambda s: "x".join(map(str, s)))
@pytest.mark.parametrize("dtype", [B.SQN_BF16, B.SQN_F16], ids=["bf16", "f16"])
def test_ragged_chunks(shape, dtype):
    import torch
    N, C, M, H, W, K, pad = shape
    rng = np.random.default_rng(sum(shape))
    tt = torch.float16 if dtype == B.SQN_F16 else torch.bfloat16
    rounded = lambda a: torch.from_numpy(np.ascontiguousarray(a, dtype=np.float32)).to(tt).float().numpy()
    x = rounded(rng.standard_normal((N, C, H, W)))
    w, b = synth.draw_conv_params(rng, C, M, K)
    w = rounded(w)
    ends = [0, N - 1]
    for inf in (False, True):           # an infinity in a tap's first layer stays with its tap: no product reaches past the last layer
        if inf:
            w[3, 0, K // 2, K // 2] = np.inf
            x[:, 0] = np.abs(x[:, 0]) + np.float32(0.5)
            x = rounded(x)
        got = G.gpu_conv(x, w, b, 1, pad, True, dtype, c_offset=8, c_total=M + 16, fill=-7.0, kernel="conv_tc").astype(np.float64)
        assert (got[:, :8] == -7.0).all() and (got[:, M + 8:] == -7.0).all()
        exp = ref.conv2d(x[ends], w, b, S=1, pad=pad, relu=True).astype(np.float64)
        wf = np.where(np.isfinite(w), w, 0)
        terms = ref.conv2d(np.abs(x[ends]), np.abs(wf), np.abs(b), S=1, pad=pad, relu=False).astype(np.float64)
        n = K * K * C + 2
        err = n * (2.0 ** -23 + 2.0 ** -24) * terms + 2.0 ** -16 * np.abs(b)[None, :, None, None]
        fin = np.isfinite(exp)
        mine = got[ends][:, 8:M + 8]
        assert fin.sum() == fin.size - (fin.size // M if inf else 0)
        np.testing.assert_array_equal(mine[~fin], exp[~fin])
        assert (np.abs(mine[fin] - exp[fin]) <= (err + ULP[dtype] * (np.abs(exp) + err) + 2.0 ** -25)[fin]).all()


@pytest.mark.parametrize("C,M,HW,K", [(512, 512, 7, 3), (384, 48, 27, 1), (64, 256, 28, 1), (256, 256, 14, 3), (112, 96, 20, 3), (96, 64, 27, 1)])
def test_only_layers_with_a_shorter_last_chunk_ask_for_it(C, M, HW, K):
    """The kernels that count MMAs per slot are slower on the layers that need not."""
    x, w, b = (B.empty_device(n, t) for n, t in (((10, HW, HW, C), B.SQN_BF16), ((M, K, K, C), B.SQN_BF16), ((M,), B.SQN_F32)))
    with G.traced() as names:
        B.conv_forward_ex(x, w, b, B.empty_device((10, HW, HW, M), B.SQN_BF16), C, M, HW, HW, K, 1, K // 2, 10, dtype=B.SQN_BF16)
    assert B.sqn_check() == B.SQN_OK
    assert len(names) == 1 and names[0].startswith("conv_tc, "), names
    assert names[0].endswith(", a shorter last chunk") == (C % 64 != 0), names
