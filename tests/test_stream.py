"""The current stream of a call without an explicit one: the raw lookup where torch has it, the
public Stream object otherwise or before CUDA is initialised."""
from types import SimpleNamespace

import pytest

from paper_2608_06628_gb300 import hybrid as H


@pytest.mark.parametrize("raw,device,up,want", [
    (lambda d: 100 + d, lambda: 3, True, 103), (lambda d: 100 + d, lambda: 3, False, 7),
    (None, lambda: 3, True, 7), (lambda d: 100 + d, None, True, 7)])
def test_current_stream(raw, device, up, want):
    c = SimpleNamespace(**{k: v for k, v in (("_cuda_getCurrentRawStream", raw), ("_cuda_getDevice", device)) if v})
    cuda = SimpleNamespace(is_initialized=lambda: up, current_stream=lambda: SimpleNamespace(cuda_stream=7))
    assert H._stream_getter(SimpleNamespace(_C=c, cuda=cuda))() == want
