"""The current stream's handle where torch has no private accessor of it."""
import types

import pytest
import torch

from paper_2404_11397_gb300 import api


@pytest.mark.parametrize("missing", ["_raw_stream", "_raw_device"])
def test_stream_handle_without_the_private_accessors(monkeypatch, missing):
    monkeypatch.setattr(api, missing, None)
    monkeypatch.setattr(torch.cuda, "current_stream", lambda: types.SimpleNamespace(cuda_stream=1234))
    assert api._stream_handle(None) == 1234
    assert api._stream_handle(types.SimpleNamespace(cuda_stream=5)) == 5
