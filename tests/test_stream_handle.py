"""The stream that a step is issued on, on the CPU: also with a torch that lacks the direct call for its handle."""
import importlib.util
import types

import pytest
import torch

from paper_2512_03416_b200 import decoder


@pytest.mark.parametrize("direct", [True, False], ids=["direct", "without"])
def test_a_step_goes_to_the_current_stream_of_its_device(direct, monkeypatch):
    if direct:
        monkeypatch.setattr(torch._C, "_cuda_getCurrentRawStream", lambda index: 100 + index, raising=False)
    else:
        monkeypatch.delattr(torch._C, "_cuda_getCurrentRawStream", raising=False)
        monkeypatch.setattr(torch.cuda, "current_stream", lambda index: types.SimpleNamespace(cuda_stream=100 + index))
    spec = importlib.util.spec_from_file_location("paper_2512_03416_b200.decoder_again", decoder.__file__)
    again = importlib.util.module_from_spec(spec)
    spec.loader.exec_module(again)
    dec = object.__new__(again.Decoder)
    dec.device = torch.device("cuda", 3)
    assert dec._stream() == 103
