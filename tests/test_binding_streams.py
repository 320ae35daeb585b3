"""Which stream the binding's calls go to: the current one, with torch's private accessors and without them, or the one given."""
import pytest
import torch

from paper_2605_16732_b200 import binding


class FakeStream:
    cuda_stream = 4711


def test_without_the_private_accessors(monkeypatch):
    monkeypatch.setattr(torch.cuda, "current_stream", lambda *a: FakeStream())
    for name in ("_raw_stream", "_current_device"):
        with monkeypatch.context() as m:
            m.setattr(binding, name, None)
            assert binding._stream() == 4711
    other = FakeStream()
    other.cuda_stream = 12
    assert binding._stream(other) == 12


@pytest.mark.gpu
def test_current_stream():
    assert binding._stream() == torch.cuda.current_stream().cuda_stream
    side = torch.cuda.Stream()
    with torch.cuda.stream(side):
        assert binding._stream() == side.cuda_stream
    assert binding._stream(side) == side.cuda_stream
