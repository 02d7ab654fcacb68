"""The Python binding's own pieces (no device)."""
from types import SimpleNamespace

import paper_2609_35099_b200 as e3j


def test_the_current_stream_is_found_with_and_without_the_raw_call(monkeypatch):
    cuda = SimpleNamespace(current_device=lambda: 3, current_stream=lambda: SimpleNamespace(cuda_stream=77))
    for c, want in ((SimpleNamespace(_cuda_getCurrentRawStream=lambda device: 10 + device), 13), (SimpleNamespace(), 77)):
        monkeypatch.setattr(e3j, "_torch_module", SimpleNamespace(_C=c, cuda=cuda))
        assert e3j._stream(None) == want
    assert e3j._stream(SimpleNamespace(cuda_stream=5)) == 5
