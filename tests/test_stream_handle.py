"""The current stream's handle, with and without torch's inner interface for it."""
import types

import pytest

from paper_2609_22441_b200 import binding as B


@pytest.mark.parametrize("handle", [0, 0x7F00])
@pytest.mark.parametrize("inner", [True, False])
def test_handle_of_the_current_stream(monkeypatch, handle, inner):
    monkeypatch.setattr(B.torch.cuda, "current_device", lambda: 3)
    monkeypatch.setattr(B.torch.cuda, "current_stream", lambda: types.SimpleNamespace(cuda_stream=handle))
    asked = []
    monkeypatch.setattr(B, "_raw_stream", (lambda device: asked.append(device) or handle) if inner else None)
    assert B._stream_ptr(None) == (handle or None)
    assert asked == ([3] if inner else [])
    assert B._stream_ptr(17) == 17
