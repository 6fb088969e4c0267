"""Sim.entropy_code's memory for the coded state, with a stand-in for the
library's call (no GPU): the bytes come back as written, the functions of
ctypes.pythonapi keep their prototypes, and an error while the memory is made
is raised as it is."""
import ctypes as C

import pytest

from paper_2302_09883_gb300 import Sim, _lib as B, sim as S


class _Library:
    def __init__(self, data):
        self.data = data

    def wcs_entropy_code_to(self, h, alloc, user, nbytes):
        nbytes._obj.value = len(self.data)
        to = alloc(None, len(self.data))
        if to:
            C.memmove(to, self.data, len(self.data))
        return 0


def _sim(monkeypatch, data):
    monkeypatch.setattr(B, "lib", lambda: _Library(data))
    return Sim.__new__(Sim)


@pytest.mark.parametrize("n", [1, 256, 6000])
def test_bytes_and_process_wide_prototypes(monkeypatch, n):
    data = bytes(k % 256 for k in range(n))
    s = _sim(monkeypatch, data)
    s.h = None
    api = (C.pythonapi.PyBytes_FromStringAndSize, C.pythonapi.PyBytes_AsString)
    before = [(f.restype, f.argtypes) for f in api]
    assert s.entropy_code() == data
    assert [(f.restype, f.argtypes) for f in api] == before


def test_an_error_in_the_callback_is_raised(monkeypatch):
    s = _sim(monkeypatch, b"abc")
    s.h = None

    def refuse(*_):
        raise OverflowError("no such size")

    monkeypatch.setattr(S, "_new_bytes", refuse)
    with pytest.raises(OverflowError):
        s.entropy_code()
