"""The current stream's handle, from torch's private functions where it has them, else its public ones."""
import sys
import types

import pytest

from paper_1609_00098_gb300 import _binding


def _torch(initialized, private):
    t = types.SimpleNamespace()
    t.cuda = types.SimpleNamespace(is_initialized=lambda: initialized,
                                   current_stream=lambda: types.SimpleNamespace(cuda_stream=0x55))
    t._C = types.SimpleNamespace()
    if private:
        t._C._cuda_getDevice = lambda: 3
        t._C._cuda_getCurrentRawStream = lambda dev: 0x1000 + dev
    return t


@pytest.mark.parametrize("initialized,private,want", [(True, True, 0x1003), (True, False, 0x55), (False, True, 0x55),
                                                      (False, False, 0x55)])
def test_current_stream(monkeypatch, initialized, private, want):
    monkeypatch.setitem(sys.modules, "torch", _torch(initialized, private))
    assert _binding._stream() == want


def test_given_streams():
    assert _binding._stream(7) == 7 and _binding._stream(types.SimpleNamespace(cuda_stream=9)) == 9
