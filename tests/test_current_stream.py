"""current_stream() while another thread makes its first call: a fake of torch's C module lets a second call in at one of the look-ups."""
import threading
import types

import pytest
import torch

from paper_1611_07151_b200 import binding as B


@pytest.mark.parametrize("raw", [True, False], ids=["raw address", "stream object"])
@pytest.mark.parametrize("at", [0, 1])
def test_first_calls_of_two_threads(monkeypatch, raw, at):
    stream = types.SimpleNamespace(cuda_stream=1234)
    monkeypatch.setattr(torch.cuda, "current_stream", lambda device=None: stream)
    monkeypatch.setattr(torch.cuda, "current_device", lambda: 0)
    seen, looked_up = [], []

    def other():
        try:
            seen.append(B.current_stream())
        except Exception as e:
            seen.append(e)

    class FakeC:
        def __getattr__(self, name):
            looked_up.append(name)
            if len(looked_up) == at + 1:
                t = threading.Thread(target=other)
                t.start()
                t.join()
            if not raw or name not in ("_cuda_getCurrentRawStream", "_cuda_getDevice"):
                raise AttributeError(name)
            return (lambda device: 1234 + device) if name == "_cuda_getCurrentRawStream" else (lambda: 0)

    monkeypatch.setattr(torch, "_C", FakeC())
    monkeypatch.setattr(B, "_raw_stream", None)
    monkeypatch.setattr(B, "_current_device", None)
    assert B.current_stream() == 1234
    assert seen and all(s == 1234 for s in seen)
