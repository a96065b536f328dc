"""The choice between the exact path's three kernels, where a wrong estimate once cost most: staged windows (strides, layer counts
that are no multiple of 4) on the tensor cores against the kernel for small layers and the FFMA kernel."""
import numpy as np
import pytest

from paper_1611_07151_b200 import binding as B
from paper_1611_07151_b200 import synth
import gpu_util as G

pytestmark = pytest.mark.gpu

# (N, Cin, Cout, H, W, K, S, pad), the kernels that may run; microseconds on the tensor cores / small / FFMA as measured
CASES = [
    ((28, 151, 53, 57, 49, 1, 3, 0), "conv_f32 ", "conv_f32_small"),        # 40 / 21 / 15
    ((46, 283, 30, 40, 26, 1, 3, 0), "conv_f32 ", "conv_f32_small"),        # 46 / 13 / 21
    ((17, 135, 68, 9, 21, 1, 1, 0), "conv_f32 ", "conv_f32_small"),         # 26 / 11 / 13
    ((13, 19, 180, 28, 50, 5, 3, 2), "conv_f32 ", "conv_f32_small"),        # 48 / 27 / 35
    ((2, 50, 65, 64, 22, 3, 1, 1), "conv_f32_small",),                      # 38 / 18 / 29
    ((19, 125, 373, 13, 11, 3, 2, 0), "conv_f32_small",),                   # 96 / 38 / 100
    ((51, 145, 6, 75, 52, 5, 1, 0), "conv_f32_tc", "conv_f32_small"),       # 1770 / 2040 / 3150
    ((50, 285, 17, 61, 56, 3, 3, 0), "conv_f32_small",),                    # 577 / 199 / 661
    ((25, 96, 16, 55, 55, 1, 1, 0), "conv_f32 "),                          # 18 / 17 / 15
    ((71, 96, 16, 55, 55, 1, 1, 0), "conv_f32 "),                          # 44 / 42 / 37
    ((8, 96, 16, 55, 55, 1, 1, 0), "conv_f32_small"),                      # - / 8.4 / 10.5
    ((19, 128, 16, 55, 55, 1, 1, 0), "conv_f32_small"),                    # - / 14 / 19
    ((116, 128, 16, 55, 55, 1, 1, 0), "conv_f32_small"),                   # - / 67 / 76
    ((16, 64, 128, 56, 56, 3, 2, 1), "conv_f32_tc",),                       # 38 / - / 65
    ((64, 3, 96, 227, 227, 7, 2, 0), "conv_f32_tc",),                       # 265 / - / 690
    ((7, 224, 40, 21, 54, 1, 1, 0), "conv_f32_small",),                     # 10.3 / 7.2 / 11.7
    ((8, 24, 40, 42, 27, 7, 1, 3), "conv_f32_small",),                      # 37 / 24 / 52
    ((12, 384, 48, 27, 27, 1, 1, 0), "conv_f32_small",),                    # 14.4 / 11.1 / 18.5
]


@pytest.mark.parametrize("case", CASES, ids=lambda c: "x".join(map(str, c[0])))
def test_the_faster_kernel_runs(case):
    (N, C, M, H, W, K, S, pad), kernels = case[0], case[1:]
    w, b = synth.draw_conv_params(np.random.default_rng(1), C, M, K)
    x = B.empty_device((N, H, W, C), B.SQN_F32).fill_(0.5)
    out = B.empty_device((N, (H + 2 * pad - K) // S + 1, (W + 2 * pad - K) // S + 1, M), B.SQN_F32)
    with G.traced() as names:
        B.conv_forward_ex(x, G.dev_w(w, B.SQN_F32), G.dev_b(b), out, C, M, H, W, K, S, pad, N, dtype=B.SQN_F32)
    assert B.sqn_check() == B.SQN_OK
    assert len(names) == 1 and names[0].startswith(kernels), names
