"""The stem and its max-pool in one launch (a forward of one image) against the oracle, on the caller's operands and on operands
packed offline.

Bound per output: exact products added to an fp32 sum that the matrix units may cut to 24 bits (2^-23 of what it holds): 224
steps on sums no larger than the sum of |kernel * input| and |bias|, the bias itself as two 16-bit numbers (2^-16 of it), the
oracle's own 148 roundings; then one rounding to the 16-bit type.  The pooled map is the maximum of the stored one, exactly."""
import numpy as np
import pytest

from oracle import ref
from paper_1611_07151_b200 import binding as B
from paper_1611_07151_b200 import synth
import gpu_util as G

pytestmark = pytest.mark.gpu
ULP = {B.SQN_BF16: 2.0 ** -8, B.SQN_F16: 2.0 ** -11}


def forward(x, params, dtype, prepacked):
    import torch
    tt = torch.float16 if dtype == B.SQN_F16 else torch.bfloat16
    names = [n for n, *_ in synth.SQUEEZENET_CONVS]
    ws = [G.dev_w(params[n][0], dtype) for n in names]
    bs = [G.dev_b(params[n][1]) for n in names]
    if prepacked:
        ws[0] = B.to_device(B.sqn_pack_stem_weights(*params["conv1"]), dtype)
    net = B.squeezenet_create(ws, bs, dtype, 1)
    if prepacked:
        B.squeezenet_set_stem_prepacked(net, True)
    xd = B.to_device(B.sqn_pack_stem_input(x), dtype) if prepacked else G.dev_act(x, dtype)
    work = torch.empty(B.squeezenet_workspace_bytes(net, 1), dtype=torch.uint8, device="cuda")
    logits = torch.empty((1, 1000), device="cuda")
    B.squeezenet_forward(net, xd, logits, None, work, 1)
    assert B.sqn_check() == B.SQN_OK
    maps = []
    for name in ("conv1", "pool1"):
        ptr, C, H, W = B.squeezenet_layer_output(net, name, work, 1)
        off = (ptr - work.data_ptr()) // 2
        maps.append(work.view(tt)[off:off + C * H * W].view(H, W, C).permute(2, 0, 1)[None].float().cpu().numpy())
    B.squeezenet_destroy(net)
    return tt, maps, logits.cpu().numpy()


@pytest.mark.parametrize("dtype,prepacked", [(B.SQN_BF16, False), (B.SQN_BF16, True), (B.SQN_F16, False)])
def test_stem_of_one_image(dtype, prepacked):
    import torch
    x, params = synth.squeezenet_case(31, 1)
    tt, (conv, pool), logits = forward(x, params, dtype, prepacked)
    rounded = lambda a: torch.from_numpy(np.ascontiguousarray(a, dtype=np.float32)).to(tt).float().numpy()
    x16, w, b = rounded(x), rounded(params["conv1"][0]), params["conv1"][1]
    exp = ref.conv2d(x16, w, b, S=2, pad=0, relu=True).astype(np.float64)
    terms = ref.conv2d(np.abs(x16), np.abs(w), np.abs(b), S=2, pad=0, relu=False).astype(np.float64)
    err = (224 * 2.0 ** -23 + 148 * 2.0 ** -24) * terms + 2.0 ** -16 * np.abs(b)[None, :, None, None]
    assert (np.abs(conv - exp) <= err + ULP[dtype] * (np.abs(exp) + err) + 2.0 ** -25).all()
    np.testing.assert_array_equal(pool, ref.maxpool(conv, 3, 2))
    if prepacked:
        np.testing.assert_array_equal(logits, forward(x, params, dtype, False)[2])
