"""How the tokens of an append are laid over the SMs (the rules compiled for the host, no GPU needed)."""
import ctypes
import os
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2607_23815_b200", "csrc")


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    gxx = shutil.which("g++") or pytest.skip("no g++")
    d = tmp_path_factory.mktemp("spread")
    (d / "shim.cpp").write_text('#include "spread.h"\n'
                                'extern "C" int prologue_tokens(int total, int sms) { return kvattn::prologue_tokens(total, sms); }\n')
    subprocess.run([gxx, "-std=c++17", "-shared", "-fPIC", f"-I{CSRC}", str(d / "shim.cpp"), "-o", str(d / "shim.so")], check=True)
    return ctypes.CDLL(str(d / "shim.so"))


@pytest.mark.parametrize("sms", [1, 2, 3, 148])                  # (1: also what is assumed where the device does not tell)
@pytest.mark.parametrize("total", [1, 2, 31, 32, 33, 147, 148, 4704, 4705, 2**31 - 1])
def test_tokens_of_a_prologue_block(lib, total, sms):
    n, others = lib.prologue_tokens(total, sms), max(sms - 1, 1)
    assert n == min(-(-total // others), 32)
