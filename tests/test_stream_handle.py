"""The stream handle of a call: the current stream's, with torch's internal raw
calls or, where a torch version lacks them, the public one."""
import types

import pytest
import torch

from paper_2304_11274_gb300 import api


@pytest.mark.parametrize("missing", ["_raw_stream", "_current_device"])
def test_without_the_internal_calls(monkeypatch, missing):
    monkeypatch.setattr(api, missing, None)
    monkeypatch.setattr(torch.cuda, "current_stream", lambda: types.SimpleNamespace(cuda_stream=7))
    assert api._stream() == 7
    assert api._stream(types.SimpleNamespace(cuda_stream=9)) == 9


@pytest.mark.gpu
def test_raw_handle_is_the_current_streams():
    assert api._stream() == torch.cuda.current_stream().cuda_stream
    s = torch.cuda.Stream()
    with torch.cuda.stream(s):
        assert api._stream() == s.cuda_stream == torch.cuda.current_stream().cuda_stream
    assert api._stream(s) == s.cuda_stream
