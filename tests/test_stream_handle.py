"""The current stream's handle comes from a short cut into PyTorch where it has
one, from the public Stream object where it has not; a given stream is used."""
import types

import pytest


@pytest.mark.parametrize("short_cut", [True, False])
def test_handle(monkeypatch, short_cut):
    import torch
    import paper_2304_05669_gb300 as F
    monkeypatch.setattr(torch.cuda, "current_device", lambda: 3)
    monkeypatch.setattr(torch.cuda, "current_stream", lambda *a: types.SimpleNamespace(cuda_stream=42))
    monkeypatch.setattr(F, "_raw_stream", (lambda device: 100 + device) if short_cut else None)
    assert F._stream() == (103 if short_cut else 42)
    assert F._stream(types.SimpleNamespace(cuda_stream=7)) == 7


@pytest.mark.gpu
def test_both_ways_agree(monkeypatch):
    import torch
    import paper_2304_05669_gb300 as F
    side = torch.cuda.Stream()
    with torch.cuda.stream(side):
        direct = F._stream()
        monkeypatch.setattr(F, "_raw_stream", None)
        assert direct == F._stream() == side.cuda_stream
