"""Band heights that the fused fire kernel chooses by the number of bands per CTA, on both sides of the rule's lines.

The height moves no sum: the values are those of a forced height, bit for bit; and the first and last image match the oracle
(fp32 sums of 16-bit operands, the squeeze map and the output rounded to bf16: 2^-8 each, the squeeze's taken through at most
a whole sum of the expands' absolute terms, here 2e-2 of the largest output)."""
import os

import numpy as np
import pytest

from oracle import ref
from paper_1611_07151_b200 import binding as B
from paper_1611_07151_b200 import synth
import gpu_util as G

pytestmark = pytest.mark.gpu
BF16 = B.SQN_BF16

# (batch, Cin, s, e, H, forced height)
CASES = [
    (16, 96, 16, 64, 55, 14),       # two bands of 4 rows per CTA
    (24, 128, 16, 64, 55, 4),       # five bands of 2 rows
    (41, 96, 16, 64, 55, 14),       # four of 4
    (120, 96, 16, 64, 55, 4),       # past the rule: the listed height
    (41, 256, 32, 128, 27, 16),     # two jobs per tile: two bands of one tile per CTA
    (90, 256, 32, 128, 27, 4),      # past the rule
    (30, 64, 16, 32, 40, 8),        # a shape that is not listed
]


@pytest.mark.parametrize("case", CASES, ids=lambda c: "x".join(map(str, c)))
def test_chosen_band_height(case):
    N, cin, s, e, H, forced = case
    x, sq, x1, x3 = synth.fire_case(sum(case), N, cin, s, e, e, H)
    dev = [G.dev_act(x, BF16), G.dev_w(sq[0], BF16), G.dev_b(sq[1]), G.dev_w(x1[0], BF16), G.dev_b(x1[1]),
           G.dev_w(x3[0], BF16), G.dev_b(x3[1])]
    scratch = B.empty_device((N, H, H, s), BF16)
    outs = []
    try:
        for band in (None, forced):
            if band:
                os.environ["SQN_FIRE_BAND"] = str(band)
            out = B.empty_device((N, H, H, 2 * e), BF16)
            out.fill_(float("nan"))
            B.fire_forward(*dev, scratch, out, cin, s, e, e, H, H, N, BF16)
            assert B.sqn_check() == B.SQN_OK
            outs.append(G.host_act(out, BF16))
    finally:
        os.environ.pop("SQN_FIRE_BAND", None)
    np.testing.assert_array_equal(outs[0], outs[1])
    ends = [0, N - 1]
    exp = ref.fire(x[ends], *sq, *x1, *x3)
    for half in (slice(0, e), slice(e, 2 * e)):
        assert G.rel_err(outs[0][ends][:, half], exp[:, half]) <= 2e-2
