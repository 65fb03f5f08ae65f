"""The binding's stream handle: torch's raw accessor, which is not a public name, or without it the public
call; both give the current stream's handle."""
import pytest
import torch

from paper_2504_02437_gb300 import api


class _Stream:
    cuda_stream = 1234


def test_without_the_raw_accessor(monkeypatch):
    monkeypatch.setattr(api, "_raw_stream", None)
    monkeypatch.setattr(torch.cuda, "current_stream", lambda *a: _Stream())
    assert api._stream() == 1234


def test_with_the_raw_accessor(monkeypatch):
    monkeypatch.setattr(api, "_raw_stream", lambda device: 100 + device)
    monkeypatch.setattr(torch.cuda, "current_device", lambda: 3)
    assert api._stream() == 103


@pytest.mark.gpu
def test_both_name_the_current_stream(monkeypatch):
    side = torch.cuda.Stream()
    for s in (torch.cuda.default_stream(), side):
        with torch.cuda.stream(s):
            with_raw = api._stream()
            with monkeypatch.context() as m:
                m.setattr(api, "_raw_stream", None)
                assert with_raw == api._stream() == s.cuda_stream
