"""The binding's stream handle where torch lacks the two private calls it takes it from (no GPU needed)."""
import types


def test_current_stream_is_the_way_back(monkeypatch):
    import torch
    from paper_1507_01009_gb300 import rv
    monkeypatch.setattr(rv, "_CURRENT", None)
    monkeypatch.setattr(torch.cuda, "init", lambda: None)
    monkeypatch.setattr(torch.cuda, "current_stream", lambda: types.SimpleNamespace(cuda_stream=0x1234))
    monkeypatch.delattr(torch._C, "_cuda_getCurrentRawStream", raising=False)
    assert rv._stream() == 0x1234
    assert rv._stream(types.SimpleNamespace(cuda_stream=0x99)) == 0x99
