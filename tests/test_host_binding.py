"""The binding's stream handle, on a stand-in for torch."""
from types import SimpleNamespace

import pytest

from paper_1112_0402_gb300 import api


def _torch(initialized, private):
    c = SimpleNamespace()
    if private:
        c._cuda_getDevice = lambda: 3
        c._cuda_getCurrentRawStream = lambda device: 1000 + device
    current = SimpleNamespace(cuda_stream=77)
    return SimpleNamespace(_C=c, cuda=SimpleNamespace(is_initialized=lambda: initialized, current_stream=lambda: current))


@pytest.mark.parametrize("initialized,private,want", [(True, True, 1003), (True, False, 77), (False, True, 77),
                                                      (False, False, 77)])
def test_current_stream(monkeypatch, initialized, private, want):
    monkeypatch.setattr(api, "_torch", _torch(initialized, private))
    assert api._stream(None) == want
    assert api._stream(SimpleNamespace(cuda_stream=5)) == 5
