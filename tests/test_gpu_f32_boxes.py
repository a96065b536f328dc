"""The exact path's tensor-core kernel on staged windows, where whole boxes of output pixels are stored by TMA: ragged maps whose last
tiles reach past the map, and the layer's slice of a wider output, against the oracle."""
import numpy as np
import pytest

from oracle import ref
from paper_1611_07151_b200 import binding as B
from paper_1611_07151_b200 import synth
import gpu_util as G
from test_gpu_f32_tensor import bound

pytestmark = pytest.mark.gpu
F32 = B.SQN_F32


@pytest.mark.parametrize("offset,total", [(8, 160), (3, 163)])      # by boxes, by 4-byte stores
@pytest.mark.parametrize("shape", [(12, 3, 96, 115, 97, 7, 2, 0), (16, 64, 128, 57, 41, 3, 2, 1), (50, 8, 100, 31, 29, 3, 2, 1),
                                   (5, 64, 64, 20, 290, 3, 1, 1)], ids=lambda s: "x".join(map(str, s)))
def test_boxes_of_pixels(shape, offset, total):
    N, C, M, H, W, K, S, pad = shape
    rng = np.random.default_rng(sum(shape))
    x = rng.standard_normal((N, C, H, W)).astype(np.float32)
    w, b = synth.draw_conv_params(rng, C, M, K)
    got = G.gpu_conv(x, w, b, S, pad, False, F32, c_offset=offset, c_total=total, fill=-7.0, kernel="conv_f32_tc box")
    assert (got[:, :offset] == -7.0).all() and (got[:, offset + M:] == -7.0).all()
    ends = [0, N - 1]
    exp = ref.conv2d(x[ends], w, b, S=S, pad=pad, relu=False)
    mine = got[ends][:, offset:offset + M].astype(np.float64)
    assert (np.abs(mine - exp) <= bound(x[ends], w, b, S, pad, K, C)).all()
    assert not np.isnan(got).any()


# (N, Cin, Cout, H, W, K, S, pad), the variant that runs: what the stores stage must not cost the kernels' source or more blocks of
# layers (microseconds with those / without)
PLANS = [((16, 3, 96, 227, 227, 7, 2, 0), "kernels packed, 1 block, 32 pixels per store"),
         ((32, 20, 256, 112, 112, 3, 2, 1), "kernels by boxes, 1 block, 16 pixels per store"),      # 246 / 104
         ((48, 18, 348, 43, 42, 3, 2, 1), "kernels by copies, 1 block, 16 pixels per store"),       # 131 / 80
         ((4, 33, 276, 29, 110, 7, 1, 3), "kernels by copies, 1 block, 16 pixels per store"),       # 339 / 237
         ((64, 20, 256, 28, 28, 5, 2, 2), "kernels by boxes, 1 block, 16 pixels per store"),        # 70 / 40
         ((20, 4, 164, 56, 53, 7, 2, 3), "kernels by boxes, 1 block, 32 pixels per store")]         # (packed, 16 pixels: 28) / 21


@pytest.mark.parametrize("shape,variant", PLANS, ids=lambda s: "x".join(map(str, s)) if isinstance(s, tuple) else s)
def test_staging_takes_nothing_from_the_plan(shape, variant):
    N, C, M, H, W, K, S, pad = shape
    rng = np.random.default_rng(sum(shape))
    x = rng.standard_normal((N, C, H, W)).astype(np.float32)
    w, b = synth.draw_conv_params(rng, C, M, K)
    got = G.gpu_conv(x, w, b, S, pad, False, F32, c_offset=8, c_total=M + 12, fill=-7.0, kernel="conv_f32_tc box, " + variant)
    assert (got[:, :8] == -7.0).all() and (got[:, 8 + M:] == -7.0).all()
    exp = ref.conv2d(x[-1:], w, b, S=S, pad=pad, relu=False)
    assert (np.abs(got[-1:, 8:8 + M].astype(np.float64) - exp) <= bound(x[-1:], w, b, S, pad, K, C)).all()
    assert not np.isnan(got).any()
