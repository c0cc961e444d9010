"""The current stream's handle: read through torch's internals where they are there, through the
public Stream object otherwise."""
from types import SimpleNamespace

import pytest

from paper_2207_10731_gb300 import binding


def _fake(initialized, internals):
    cuda = SimpleNamespace(is_initialized=lambda: initialized,
                           current_stream=lambda: SimpleNamespace(cuda_stream=77))
    c = SimpleNamespace(_cuda_getDevice=lambda: 3, _cuda_getCurrentRawStream=lambda d: 100 + d)
    return SimpleNamespace(cuda=cuda, _C=c if internals else SimpleNamespace())


@pytest.mark.parametrize("initialized,internals,want", [(True, True, 103), (True, False, 77),
                                                        (False, True, 77), (False, False, 77)])
def test_current_stream(monkeypatch, initialized, internals, want):
    monkeypatch.setattr(binding, "_torch_mod", _fake(initialized, internals))
    assert binding._stream_ptr(None) == want
    assert binding._stream_ptr(SimpleNamespace(cuda_stream=5)) == 5
