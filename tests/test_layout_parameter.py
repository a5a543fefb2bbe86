"""A Layout stands for its handle in any ctypes call, whether or not the called
function has declared its argument types (an undeclared integer argument would
be passed as a 32-bit int). CPU only: a made-up handle, never dereferenced."""

import ctypes

import pytest

from paper_2607_02893_gb300.vbq import Layout

HANDLE = 0x7F12_3456_7890


@pytest.fixture
def layout():
    lay = Layout(HANDLE, 1, 64)
    yield lay
    lay.handle = None                 # nothing to free


def test_without_declared_argument_types(layout):
    f = ctypes.CDLL(None).llabs       # long long -> long long
    f.restype = ctypes.c_longlong
    assert f(layout) == HANDLE


def test_with_declared_argument_types(layout):
    f = ctypes.CDLL(None).llabs
    f.restype, f.argtypes = ctypes.c_longlong, [ctypes.c_void_p]
    assert f(layout) == HANDLE
    assert (ctypes.c_void_p * 1)(layout._as_parameter_)[0] == HANDLE


def test_freed_layout_is_refused(layout):
    f = ctypes.CDLL(None).llabs
    f.restype, f.argtypes = ctypes.c_longlong, [ctypes.c_void_p]
    layout.handle = None
    with pytest.raises(ValueError):
        layout._as_parameter_
    with pytest.raises((ValueError, ctypes.ArgumentError)):
        f(layout)
