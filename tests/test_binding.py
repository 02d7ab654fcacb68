"""The Python binding's own pieces (no device)."""
from types import SimpleNamespace

import paper_2609_35099_b200 as e3j


def test_the_current_stream_is_found_with_and_without_the_raw_calls():
    cuda = SimpleNamespace(current_stream=lambda: SimpleNamespace(cuda_stream=77))
    raw = dict(_cuda_getCurrentRawStream=lambda device: 10 + device, _cuda_getDevice=lambda: 3)
    for calls, want in ((raw, 13), ({}, 77), ({"_cuda_getDevice": raw["_cuda_getDevice"]}, 77)):
        assert e3j._stream_reader(SimpleNamespace(_C=SimpleNamespace(**calls), cuda=cuda))() == want
    assert e3j._stream(SimpleNamespace(cuda_stream=5)) == 5
