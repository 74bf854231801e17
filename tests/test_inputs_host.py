"""Which input arrays a kernel reads in place (csrc/gm_inputs.h, compiled for the host):
those in the context's own device's memory, at an address its loads can use."""
import ctypes as C
import os
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))),
                    "paper_1708_09705_gb300", "csrc")


@pytest.fixture(scope="module")
def in_place(tmp_path_factory):
    cxx = shutil.which("g++") or shutil.which("c++")
    if not cxx:
        pytest.skip("no C++ compiler")
    d = tmp_path_factory.mktemp("inputs")
    (d / "h.cpp").write_text('#include "gm_inputs.h"\nextern "C" int f(int a, int b, const void* p, '
                             'size_t n) { return gm::read_in_place(a, b, p, n); }\n')
    subprocess.run([cxx, "-shared", "-fPIC", "-std=c++17", f"-I{CSRC}", str(d / "h.cpp"), "-o",
                    str(d / "h.so")], check=True)
    f = C.CDLL(str(d / "h.so")).f
    f.argtypes = [C.c_int, C.c_int, C.c_void_p, C.c_size_t]
    return f


@pytest.mark.parametrize("device,ctx,address,want", [
    (0, 0, 0x7000, 1), (1, 1, 0x7008, 1),
    (1, 0, 0x7000, 0), (0, 1, 0x7000, 0),        # another GPU's memory
    (-1, 0, 0x7000, 0),                          # host, managed, unknown
    (0, 0, 0x7004, 0), (0, 0, 0x7001, 0)])       # misaligned for doubles
def test_read_in_place(in_place, device, ctx, address, want):
    assert in_place(device, ctx, address, 8) == want
