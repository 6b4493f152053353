"""The binding's current stream: the raw handle where torch has it, the public call where it has not."""
import types

import pytest


@pytest.mark.parametrize("raw", [True, False])
def test_current_stream_with_and_without_the_raw_handle(raw, monkeypatch):
    import torch
    from paper_2512_14090_b200 import build
    build.build()
    from paper_2512_14090_b200 import binding
    monkeypatch.setattr(torch.cuda, "current_stream", lambda device=None: types.SimpleNamespace(cuda_stream=1000 + (device or 0)))
    monkeypatch.setattr(torch.cuda, "current_device", lambda: 3)
    if raw:
        monkeypatch.setattr(torch._C, "_cuda_getCurrentRawStream", lambda device: 2000 + device, raising=False)
    else:
        monkeypatch.delattr(torch._C, "_cuda_getCurrentRawStream", raising=False)
    monkeypatch.setattr(binding, "_raw_stream", None)
    assert binding._stream() == (2003 if raw else 1003)
    assert binding._stream(types.SimpleNamespace(cuda_stream=7)) == 7
