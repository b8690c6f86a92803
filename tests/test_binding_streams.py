"""CPU: the stream handle that the binding passes on."""
import torch

from paper_2301_01719_gb300 import api


class Stream:
    cuda_stream = 0x1234


def test_the_current_stream_with_and_without_torchs_raw_call(monkeypatch):
    dev = torch.device("cuda", 3)
    asked = []

    def raw(index):
        asked.append(index)
        return 0x77

    monkeypatch.setattr(api, "_raw_stream", raw)
    assert api._stream(None, dev) == 0x77 and asked == [3]
    monkeypatch.setattr(api, "_raw_stream", None)
    monkeypatch.setattr(torch.cuda, "current_stream", lambda d: asked.append(d) or Stream())
    assert api._stream(None, dev) == 0x1234 and asked[-1] == dev


def test_a_given_stream_is_passed_on():
    dev = torch.device("cuda", 0)
    assert api._stream(Stream(), dev) == 0x1234
    assert api._stream(0x55, dev) == 0x55 and api._stream(0, dev) == 0
