"""How the tokens of an append are laid over the SMs (the rules compiled for the host, no GPU needed)."""
import ctypes
import os
import re
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2607_23815_b200", "csrc")


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    gxx = shutil.which("g++") or pytest.skip("no g++")
    d = tmp_path_factory.mktemp("spread")
    (d / "shim.cpp").write_text('#include "spread.h"\n'
                                'extern "C" void append_spread(int total, int chunks, int sms, int* r) {\n'
                                '  const kvattn::AppendSpread a = kvattn::append_spread(total, chunks, sms);\n'
                                '  r[0] = a.blocks; r[1] = a.warps; r[2] = a.smem; r[3] = a.smem_front;\n}\n'
                                'static std::atomic<bool> done[4]; static int calls;\n'
                                'extern "C" int once(int device, int works) {\n'
                                '  return kvattn::once_per_device(done, device, [&] { ++calls; return works != 0; }) + 10 * calls;\n}\n'
                                'extern "C" int prologue_tokens(int total, int sms) { return kvattn::prologue_tokens(total, sms); }\n')
    subprocess.run([gxx, "-std=c++17", "-shared", "-fPIC", f"-I{CSRC}", str(d / "shim.cpp"), "-o", str(d / "shim.so")], check=True)
    return ctypes.CDLL(str(d / "shim.so"))


@pytest.mark.parametrize("sms", [1, 2, 3, 148])                  # (1: also what is assumed where the device does not tell)
@pytest.mark.parametrize("total", [1, 2, 31, 32, 33, 147, 148, 4704, 4705, 2**31 - 1])
def test_tokens_of_a_prologue_block(lib, total, sms):
    n, others = lib.prologue_tokens(total, sms), max(sms - 1, 1)
    assert n == min(-(-total // others), 32)


def _fit(smem):
    return 228 * 1024 // (smem + 1024)                           # blocks of that much shared memory on an SM


def _spread(lib, total, chunks, sms):
    r = (ctypes.c_int * 4)()
    lib.append_spread(total, chunks, sms, r)
    return list(r)


def _totals(sms):
    return sorted(({1, 2, 3, 37} | {k * sms + d for k in range(1, 26) for d in (-1, 0, 1)} | {sms // 2, sms // 2 + 1}) - {0})


@pytest.mark.parametrize("chunks", [8, 63, 64, 127, 128, 129, 512])
@pytest.mark.parametrize("sms", [1, 147, 148])
def test_every_token_has_a_warp_and_no_sm_more_than_its_share(lib, sms, chunks):
    most = 8 if chunks < 64 else 24 if chunks <= 128 else 16
    for total in _totals(sms):
        blocks, warps, smem, front = _spread(lib, total, chunks, sms)
        share = -(-total // sms)
        assert (blocks == 0) == (share > most)
        if blocks == 0:
            continue
        n = _fit(smem)
        assert (blocks - 1) * warps < total <= blocks * warps and 1 <= warps <= 8
        assert blocks <= n * sms                                 # all of them are resident at once
        k = -(-share // 8)                                       # blocks of an SM
        assert k * warps < share + k and n in (k, 2 * k)         # an SM's share, rounded up to whole blocks, where n is k


@pytest.mark.parametrize("chunks", [8, 64, 128, 512])
def test_a_second_call_finds_room_beside_the_first(lib, chunks, sms=148):
    for total in _totals(sms):
        blocks, _, smem, front = _spread(lib, total, chunks, sms)
        if 0 < blocks <= sms:
            assert 2 * blocks <= _fit(front) * sms, total
            if total <= sms or chunks < 128:                     # (larger appends of 4 KB rows keep an SM per block)
                assert 2 * blocks <= _fit(smem) * sms, total


def test_a_device_without_the_opt_in_goes_without(lib):
    # (result + 10 x calls so far) a device that is not in the table, one where it fails, then works, then is remembered
    assert [lib.once(-1, 1), lib.once(4, 1), lib.once(2, 0), lib.once(2, 0), lib.once(2, 1), lib.once(2, 0), lib.once(3, 0)] == [0, 0, 10, 20, 31, 31, 40]


@pytest.mark.parametrize("name", ["pool.cu", "attn_extend_tc.cu"])
def test_the_opt_in_is_asked_for_the_kernel_that_is_launched(name):
    text = open(os.path.join(CSRC, name)).read()
    found = re.findall(r"static std::atomic<bool> allowed\[kMaxDevices\];\s*if \(sp\.blocks > 0 && allow_smem\(\(const void\*\)([^,]+),[^;]*?"
                       r"launch_early\(([^,]+),[^;]*sp\.blocks", text)
    assert found and all(a == b for a, b in found) and len(found) == text.count("allow_smem(")
