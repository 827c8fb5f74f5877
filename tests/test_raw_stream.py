"""The stream a call runs on: the caller's, else torch's current one, with or
without torch's private function that gives it as a number.
"""

import types

import pytest

torch = pytest.importorskip("torch")

from paper_1310_7297_gb300 import vcm


def test_current_stream_with_and_without_the_private_call(monkeypatch):
    dev = torch.device("cuda", 1)
    monkeypatch.setattr(torch.cuda, "current_stream", lambda d=None: types.SimpleNamespace(cuda_stream=70 + d.index))
    monkeypatch.setattr(torch._C, "_cuda_getCurrentRawStream", lambda index: 40 + index, raising=False)
    assert vcm._raw_stream(None, dev) == 41
    monkeypatch.delattr(torch._C, "_cuda_getCurrentRawStream")
    assert vcm._raw_stream(None, dev) == 71
    assert vcm._raw_stream(types.SimpleNamespace(cuda_stream=5), dev) == 5
