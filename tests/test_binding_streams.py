"""The stream a call goes to: a given stream or handle as it is, else the current
stream, also where torch has no raw handle of it to give."""
import types

import pytest
import torch

from paper_2609_13141_gb300 import sas


@pytest.mark.parametrize("raw", [True, False])
def test_current_stream_with_and_without_the_raw_handle(monkeypatch, raw):
    monkeypatch.setattr(torch.cuda, "current_device", lambda: 3)
    monkeypatch.setattr(torch.cuda, "current_stream", lambda: types.SimpleNamespace(cuda_stream=0x1234))
    monkeypatch.setattr(sas, "_raw_stream", (lambda dev: 0x1234 if dev == 3 else 0) if raw else None)
    assert sas._stream(None).value == 0x1234


def test_given_streams():
    assert sas._stream(types.SimpleNamespace(cuda_stream=0x88)).value == 0x88
    assert sas._stream(0x99).value == 0x99


@pytest.mark.gpu
def test_raw_handle_is_the_current_streams():
    s = torch.cuda.Stream()
    with torch.cuda.stream(s):
        assert sas._stream(None).value == s.cuda_stream
