"""The calls that the binding makes through plain integers (csrc/calls.cpp): status codes of the C ABI come back, wrong arguments
raise, nothing touches a device.  Where the module was not built the same calls go through ctypes."""
import ctypes as C
import os
import subprocess
import sys

import pytest

from paper_2311_14272_b200 import binding as B
from paper_2311_14272_b200 import build as build_mod


@pytest.fixture(scope="module")
def native():
    build_mod.build()
    B.load()
    return B._native


def test_status_codes_come_back(native):
    assert native.spmm(0, 1, 8, 8, 1, 8, 0, 0) == B.INVALID_ARG
    assert native.spmm_conv(0, 1, 1, 8, 8, 64, 3, 3, 1, 0, 1, 8, 0, 0) == B.INVALID_ARG
    assert native.spmm_conv(0, 1, 1, 2 ** 33, 8, 64, 3, 3, 1, 0, 1, 8, 0, 0) == B.BAD_SHAPE        # not an int32
    assert native.decode(0, 1, 8, 0) == B.INVALID_ARG
    assert native.encode_sizes(0) == (B.INVALID_ARG, 0, 0)
    assert native.encode(256, 8, 0, 256, 256, 0, 0) == (B.INVALID_ARG, 0)
    desc = B.make_desc(64, 128, 2, 5, 32, 32, 0.5)
    assert native.build_mask(256, 128, C.addressof(desc), 256, 256, 0, 0) == (B.UNSUPPORTED, 0)


@pytest.mark.parametrize("name,count", [("spmm", 8), ("spmm_conv", 14), ("decode", 4), ("build_mask", 7), ("encode_sizes", 1), ("encode", 7)])
def test_wrong_arguments_raise(native, name, count):
    call = getattr(native, name)
    with pytest.raises(TypeError):
        call(*[0] * (count - 1))
    with pytest.raises(TypeError):
        call(*[0] * (count + 1))
    with pytest.raises(TypeError):
        call(*[0] * (count - 1), None)
    with pytest.raises(OverflowError):
        call(*[0] * (count - 1), 2 ** 70)


def test_layers_are_released_together():
    masks, handles = (C.c_void_p * 3)(), (C.c_void_p * 3)()
    B.crisp_destroy_layers(masks, handles)                 # nothing in them: nothing to do
    assert B.load().crisp_destroy_layers(-1, masks, handles) == B.INVALID_ARG
    assert B.load().crisp_destroy_layers(1, None, handles) == B.INVALID_ARG


def test_the_library_loads_without_the_module():
    """In a process that cannot import _calls: the same calls, arguments and results through ctypes."""
    code = """
import ctypes as C, sys
sys.modules["paper_2311_14272_b200._calls"] = None           # an import of it fails
from paper_2311_14272_b200 import binding as B
B.load()
n = B._native
assert type(n).__name__ == "_CtypesCalls"
assert n.spmm(0, 1, 8, 8, 1, 8, 0, 0) == B.INVALID_ARG
assert n.spmm_conv(0, 1, 1, 8, 8, 64, 3, 3, 1, 0, 1, 8, 0, 0) == B.INVALID_ARG
assert n.spmm_conv(0, 1, 1, 2 ** 33, 8, 64, 3, 3, 1, 0, 1, 8, 0, 0) == B.BAD_SHAPE
assert n.decode(0, 1, 8, 0) == B.INVALID_ARG
assert n.encode_sizes(0) == (B.INVALID_ARG, 0, 0)
assert n.encode(256, 8, 0, 256, 256, 0, 0) == (B.INVALID_ARG, 0)
desc = B.make_desc(64, 128, 2, 5, 32, 32, 0.5)
assert n.build_mask(256, 128, C.addressof(desc), 256, 256, 0, 0) == (B.UNSUPPORTED, 0)
print("loaded")
"""
    root = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
    out = subprocess.run([sys.executable, "-c", code], cwd=root, capture_output=True, text=True, timeout=300)
    assert out.returncode == 0 and "loaded" in out.stdout, out.stderr
