"""Which host buffers attn_extend_host lets a kernel copy: those that lie in one pinned range from the first byte to the last
(compiled for the host, no GPU needed)."""
import ctypes
import os
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2607_23815_b200", "csrc")


@pytest.fixture(scope="module")
def view(tmp_path_factory):
    gxx = shutil.which("g++") or pytest.skip("no g++")
    d = tmp_path_factory.mktemp("host_view")
    (d / "shim.cpp").write_text('#include "host_view.h"\nextern "C" uintptr_t view(int pinned, uintptr_t device, uintptr_t start, size_t size, size_t bytes) {\n'
                                "  return kvattn::device_view(kvattn::HostAddress{pinned != 0, device, start, size}, bytes);\n}\n")
    subprocess.run([gxx, "-std=c++17", "-shared", "-fPIC", f"-I{CSRC}", str(d / "shim.cpp"), "-o", str(d / "shim.so")], check=True)
    f = ctypes.CDLL(str(d / "shim.so")).view
    f.restype, f.argtypes = ctypes.c_size_t, [ctypes.c_int] + [ctypes.c_size_t] * 4
    # registrations (start, bytes); an address outside all of them is not pinned
    def at(regs, address, n):
        for start, size in regs:
            if start <= address < start + size:
                return f(1, address, start, size, n)
        return f(0, 0, 0, 0, n)
    return at


def test_one_range(view):
    r = [(0x10000, 0x4000)]
    assert view(r, 0x10000, 0x4000) == 0x10000 and view(r, 0x13FFC, 4) == 0x13FFC and view(r, 0x10004, 8) == 0x10004
    assert view(r, 0x10000, 0x4001) == 0 and view(r, 0x13FFC, 5) == 0 and view(r, 0x20000, 4) == 0
    assert view(r, 0x10002, 4) == 0                              # the kernel moves whole words


def test_two_registrations_with_a_gap_between_them(view):
    r = [(0x10000, 0x1000), (0x12000, 0x1000)]                   # the first and the last byte of the buffer are both pinned
    assert view(r, 0x10800, 0x2000) == 0
    assert view(r, 0x10800, 0x800) == 0x10800 and view(r, 0x12800, 0x800) == 0x12800


def test_the_library_asks_for_the_range():
    text = open(os.path.join(CSRC, "api.cu")).read()
    assert "RANGE_START_ADDR" in text and "RANGE_SIZE" in text and "kvattn::device_view(" in text
