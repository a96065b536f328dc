"""The C marshalling of conv_forward_ex and fire_forward hands the library what ctypes hands it: a recording function in the library's
place, and the arguments that are left to ctypes."""
import ctypes

import numpy as np
import pytest
import torch

from paper_1611_07151_b200 import binding as B

pytestmark = pytest.mark.skipif(B._native is None, reason="marshalling module not built")
CONV = ctypes.CFUNCTYPE(ctypes.c_int, *([ctypes.c_void_p] * 4 + [ctypes.c_int] * 8 + [ctypes.POINTER(B.sqn_conv_opts)]))
FIRE = ctypes.CFUNCTYPE(ctypes.c_int, *([ctypes.c_void_p] * 9 + [ctypes.c_int] * 8 + [ctypes.c_void_p]))


class Lib:
    """Stands in for the loaded library: both paths end in the same recording functions."""

    def __init__(self, status=0):
        self.seen = []

        def conv(*a):
            o = a[12].contents
            self.seen.append(a[:12] + tuple(getattr(o, n) for n, _ in B.sqn_conv_opts._fields_))
            return status

        def fire(*a):
            self.seen.append(a)
            return status

        self.conv_forward_ex, self.fire_forward = CONV(conv), FIRE(fire)
        self.sqn_status_string = lambda rc: b"status"


@pytest.fixture(params=[0, -2])
def fake(monkeypatch, request):
    lib = Lib(request.param)
    monkeypatch.setattr(B, "_lib", lib)
    monkeypatch.setattr(B, "_conv_forward_ex_at", ctypes.cast(lib.conv_forward_ex, ctypes.c_void_p).value)
    monkeypatch.setattr(B, "_fire_forward_at", ctypes.cast(lib.fire_forward, ctypes.c_void_p).value)
    monkeypatch.setattr(B, "current_stream", lambda: 0x7f0000001234)
    lib.status = request.param
    return lib


def both(fake, monkeypatch, call):
    results = []
    for native in (B._native, None):
        monkeypatch.setattr(B, "_native", native)
        try:
            results.append(call())
        except Exception as e:
            results.append((type(e), str(e)))
    assert results[0] == results[1], results
    return results[0]


t = torch.arange(64, dtype=torch.float32)
BIG = 0xffff800012345670                       # (addresses with the top bit set)


@pytest.mark.parametrize("args,kw", [
    ((t, t[4:], t[8:], t[12:], 3, 4, 5, 6, 7, 1, 0, 2), {}),
    ((BIG, None, 16, t, 3, 4, 5, 6, 7, 1, -1, 2), dict(dtype=2, relu=0, out_c_offset=8, out_c_total=96, stream=0, workspace=t, workspace_bytes=1 << 40)),
    ((t, t, t, t, True, 4, 5, 6, 7, 1, 0, 2), dict(relu=[], fuse_maxpool="yes", fuse_global_avgpool=None, stream=BIG)),
    ((t.numpy(), t, t.numpy(), t, 3, 4, 5, 6, 7, 1, 0, 2), dict(workspace=t.numpy())),        # left to ctypes, like the following ones
    ((t, t, t, t, 1 << 40, 4, 5, 6, 7, 1, 0, 2), {}),
    ((t, t, t, t, 3, 4, 5, 6, 7, 1, 0, 2), dict(stream=ctypes.c_void_p(77))),
    ((t, t, t, t, 3.5, 4, 5, 6, 7, 1, 0, 2), {}),
    ((t, "nothing", t, t, 3, 4, 5, 6, 7, 1, 0, 2), {}),
    ((t, t, t, t, 3, 4, 5, 6, 7, 1, 0, 2), dict(workspace_bytes=1.5)),
])
def test_convolution(fake, monkeypatch, args, kw):
    result = both(fake, monkeypatch, lambda: B.conv_forward_ex(*args, **kw))
    assert len(fake.seen) in (0, 2)
    assert len(fake.seen) == 0 or fake.seen[0] == fake.seen[1]
    if fake.seen:
        assert result is None if fake.status == 0 else result[0] is B.SqnError


@pytest.mark.parametrize("args,kw", [
    ((t, t[4:], t, t[8:], t, t, t, t, t, 96, 16, 64, 64, 55, 54, 1, 1), {}),
    ((t, t, t, t, t, t, BIG, None, t, 96, 16, 64, 64, 55, 54, 1, 1), dict(stream=0)),
    ((t, t, t, t, t.numpy(), t, t, t, t, 96, 16, 64, 64, 55, 54, 1, 1), {}),
    ((t, t, t, t, t, t, t, t, t, 96, np.int64(16), 64, 64, 55, 54, 1, 1), {}),
])
def test_fire_layer(fake, monkeypatch, args, kw):
    both(fake, monkeypatch, lambda: B.fire_forward(*args, **kw))
    assert len(fake.seen) in (0, 2)
    assert len(fake.seen) == 0 or fake.seen[0] == fake.seen[1]
