"""The current stream's handle, as the binding asks torch for it: with torch's
internal functions, and in a version without them (no GPU needed)."""
from types import SimpleNamespace

import pytest


def torch_with(**internal):
    streams = {0: 100, 1: 101}
    torch = SimpleNamespace(device=0, calls=0)

    def current_stream():
        torch.calls += 1
        return SimpleNamespace(cuda_stream=streams[torch.device])

    have = {"_cuda_getDevice": lambda: torch.device, "_cuda_getCurrentRawStream": lambda d: streams[d]}
    torch._C = SimpleNamespace(**{k: v for k, v in have.items() if internal.get(k, True)})
    torch.cuda = SimpleNamespace(current_stream=current_stream)
    return torch


@pytest.mark.parametrize("internal", [{}, {"_cuda_getDevice": False}, {"_cuda_getCurrentRawStream": False},
                                      {"_cuda_getDevice": False, "_cuda_getCurrentRawStream": False}])
def test_current_stream_with_and_without_internals(monkeypatch, internal):
    from paper_cs_0404008_gb300 import gfpdot as g
    torch = torch_with(**internal)
    monkeypatch.setattr(g, "_torch", torch)
    monkeypatch.setattr(g, "_raw_stream", None)
    assert [g._stream(None) for _ in range(3)] == [100] * 3
    torch.device = 1                       # the current device's stream, each time
    assert [g._stream(None) for _ in range(2)] == [101] * 2
    assert torch.calls == (5 if internal else 1)
    assert g._stream(7) == 7 and g._stream(SimpleNamespace(cuda_stream=8)) == 8
