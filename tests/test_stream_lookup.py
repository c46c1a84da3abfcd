"""The stream that a call without one goes to: torch's current one, whichever way it is read."""
import sys
from types import SimpleNamespace

import pytest

from paper_1809_07726_gb300 import cphremd


def _torch(internals):
    return SimpleNamespace(cuda=SimpleNamespace(is_available=lambda: True,
                                                current_stream=lambda: SimpleNamespace(cuda_stream=77)),
                           _C=internals)


@pytest.mark.parametrize("internals", [
    SimpleNamespace(),
    SimpleNamespace(_cuda_getCurrentRawStream=lambda d: 77),
    SimpleNamespace(_cuda_getCurrentRawStream=lambda d: 77 if d == 3 else 0, _cuda_getDevice=lambda: 3)])
def test_current_stream_with_and_without_the_short_reads(monkeypatch, internals):
    monkeypatch.setitem(sys.modules, "torch", _torch(internals))
    monkeypatch.setattr(cphremd, "_raw_stream", None)
    assert [cphremd._stream(None) for _ in range(3)] == [77] * 3
    assert cphremd._stream(5) == 5 and cphremd._stream(0) == 0
