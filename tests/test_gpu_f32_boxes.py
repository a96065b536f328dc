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
