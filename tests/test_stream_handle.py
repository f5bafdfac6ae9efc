"""The current stream's handle, where torch has the functions that give it
without a Stream object and where it has them not (no GPU: both are faked)."""
from __future__ import annotations

import types

import pytest


@pytest.mark.parametrize("missing", [None, "_cuda_getCurrentRawStream", "_cuda_getDevice"])
def test_current_stream_is_followed(monkeypatch, missing):
    import torch
    from paper_2604_21117_gb300 import build_lib
    build_lib.build()
    from paper_2604_21117_gb300 import btree
    current = {"device": 0, "streams": {0: 111, 1: 222}}
    monkeypatch.setattr(btree, "_raw_stream", None)
    monkeypatch.setattr(btree, "_current_device", None)
    monkeypatch.setattr(torch.cuda, "current_stream",
                        lambda: types.SimpleNamespace(cuda_stream=current["streams"][current["device"]]))
    monkeypatch.setattr(torch._C, "_cuda_getCurrentRawStream", lambda d: current["streams"][d], raising=False)
    monkeypatch.setattr(torch._C, "_cuda_getDevice", lambda: current["device"], raising=False)
    if missing:
        monkeypatch.delattr(torch._C, missing)
    assert [btree._stream_handle(None) for _ in range(2)] == [111, 111]
    current["streams"][0] = 333  # another current stream
    assert btree._stream_handle(None) == 333
    current["device"] = 1  # another device
    assert btree._stream_handle(None) == 222
    assert btree._stream_handle(7) == 7 and btree._stream_handle(types.SimpleNamespace(cuda_stream=9)) == 9
