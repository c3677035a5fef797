"""torch's default stream has the handle 0, which the C ABI takes for "a new stream"."""
from types import SimpleNamespace

from paper_1411_3212_gb300 import mqr


def test_default_stream_is_named_explicitly():
    assert mqr._handle(SimpleNamespace(cuda_stream=0)) == 1          # cudaStreamLegacy
    assert mqr._handle(SimpleNamespace(cuda_stream=0x7f00)) == 0x7f00
