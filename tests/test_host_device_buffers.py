"""The buffers a network keeps between calls (csrc/devbuf.h), over a fake of
the CUDA calls: what a captured graph refers to outlives later growth, and
nothing else piles up."""
import ctypes as C
import os
import shutil
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)


@pytest.fixture
def buf(tmp_path):
    gxx = shutil.which(os.environ.get("CXX", "g++"))
    nvcc = shutil.which(os.environ.get("NVCC", "nvcc"))
    if gxx is None or nvcc is None:
        pytest.skip("no compiler")
    cuda = os.path.join(os.path.dirname(os.path.dirname(os.path.realpath(nvcc))), "include")
    out = str(tmp_path / "libdevbuf.so")
    subprocess.check_call([gxx, "-O1", "-std=c++17", "-shared", "-fPIC",
                           # the fakes, whatever the process has loaded
                           "-Wl,-Bsymbolic", "-I", cuda,
                           os.path.join(HERE, "host", "device_buffers.cpp"), "-o", out])
    lib = C.CDLL(out)
    lib.buf_call.argtypes = [C.c_size_t, C.c_int, C.c_int]
    lib.buf_call.restype = C.c_void_p
    lib.buf_live.argtypes = [C.c_void_p]
    return lib


def test_a_captured_buffer_outlives_growth(buf):
    a = buf.buf_call(100, 0, 0)              # the warm-up call
    assert buf.buf_call(100, 1, 0) == a      # the capture
    b = buf.buf_call(1000, 0, 0)             # a larger call: the graph still replays
    assert b != a and buf.buf_live(a) and buf.buf_live(b)
    assert buf.buf_call(50, 0, 0) == b
    assert buf.buf_call(500, 1, 0) == b      # a second capture, in the new buffer
    c = buf.buf_call(2000, 0, 0)
    assert buf.buf_live(a) and buf.buf_live(b) and buf.buf_live(c) and buf.buf_count() == 3


def test_other_buffers_are_given_back(buf):
    a = buf.buf_call(100, 0, 0)
    for need in (200, 300, 400):
        b = buf.buf_call(need, 0, 0)
        assert buf.buf_count() == 1 and buf.buf_live(b)
    del a
    assert buf.buf_call(10**6, 0, 1) is None          # no memory
    assert buf.buf_call(100, 0, 0) is not None and buf.buf_count() == 1
