"""The native half of the binding checks its arguments before it calls the library (no GPU needed)."""
import os
import subprocess
import sys

import numpy as np
import pytest
import torch

from paper_2607_23815_b200 import build, kvattn

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


class _NoPool:
    ptr = None


def test_tensors_must_be_contiguous_and_on_the_gpu():
    t, i = torch.zeros(2, 4, 64, dtype=torch.bfloat16), torch.zeros(2, 8, dtype=torch.int32)
    dec = lambda q: kvattn.attn_decode(_NoPool, q, i, i[0], 5, 1.0, t, t, None, 0)
    with pytest.raises(AssertionError, match="CUDA"):
        dec(t)
    with pytest.raises(AssertionError, match="contiguous"):
        dec(t.transpose(0, 1))
    with pytest.raises(TypeError, match="torch tensor"):
        dec([1, 2])


def test_errors_of_the_library_come_back_as_kverror():
    with pytest.raises(kvattn.KvError) as e:                              # no pool: refused by the library itself
        kvattn.attn_mixed(_NoPool, 8, 1.0, None, None, None, 0)
    assert e.value.status == kvattn.KV_ERR_INVALID
    with pytest.raises(TypeError):                                        # a structure of another kind
        kvattn.attn_mixed(_NoPool, 8, 1.0, kvattn.DecodeArgs(), None, None, 0)


_NO_STORAGE = """
import faulthandler; faulthandler.enable()
import torch
from torch._subclasses.fake_tensor import FakeTensorMode
from paper_2607_23815_b200 import build, kvattn
class NoPool:
    ptr = None
with FakeTensorMode():
    args = [torch.empty(3, 2, 4, 64, dtype=torch.bfloat16, device="cuda"), torch.empty(3, 2, 8, dtype=torch.int32, device="cuda"),
            torch.empty(3, 64, dtype=torch.uint8, device="cuda")]
calls = {
    "append": lambda t, i, b: kvattn.kv_append(NoPool, t, None, None, i, None, i, 0),
    "decode": lambda t, i, b: kvattn.attn_decode(NoPool, t, i, None, 5, 1.0, None, None, None, 0),
    "extend": lambda t, i, b: kvattn.attn_extend(NoPool, t, None, i, i, None, 1, 5, 1.0, None, None, None, 0),
    "planned": lambda t, i, b: kvattn.attn_extend_planned(NoPool, t, None, i, i, None, 1, 5, 1.0, None, None, None, 0),
    "extend_append": lambda t, i, b: kvattn.attn_extend_append(NoPool, t, None, None, None, i, i, None, 1, 5, 1.0, None, None, None, 0),
    "plan": lambda t, i, b: kvattn.attn_extend_plan(NoPool, 4, None, i, i, None, 2, 1, 5, None, 0),
    "shared": lambda t, i, b: kvattn.attn_extend_shared(NoPool, t, None, None, i, i, i, i, 1, 1, 5, 1.0, None, None, None, 0),
    "mixed": lambda t, i, b: kvattn.attn_mixed(NoPool, 4, 1.0, None, None, b, 0),
}
def refused(*tensors):
    for name, call in calls.items():
        for _ in range(3):
            try:
                call(*tensors)
            except RuntimeError as e:
                assert not isinstance(e, kvattn.KvError), name
            else:
                raise SystemExit(name + ": no error")
    return tensors[0]
torch.vmap(refused)(*args)
print("all refused")
"""


def test_tensors_without_storage_are_an_error_and_not_a_crash():
    # the address of such a tensor (here: one that vmap batches) cannot be had; the exception must not leave the call without
    # the interpreter lock
    r = subprocess.run([sys.executable, "-c", _NO_STORAGE], capture_output=True, text=True, cwd=ROOT, timeout=300)
    assert r.returncode == 0 and "all refused" in r.stdout, (r.returncode, r.stdout, r.stderr[-2000:])


def _host_call(out, stream=0):
    t, i = torch.zeros(2, 4, 64, dtype=torch.bfloat16), torch.zeros(2, 8, dtype=torch.int32)
    with pytest.raises(kvattn.KvError) as e:                              # no pool: refused by the library itself
        kvattn.attn_extend_host(_NoPool, t, t, t, i[0], i, i[0], i[0], 1, 5, 1.0, out, torch.zeros(2, 4), None, stream)
    assert e.value.status == kvattn.KV_ERR_INVALID


def test_results_go_to_the_tensor_s_own_memory():
    base = torch.zeros(2, 4, 64, dtype=torch.bfloat16)
    out = torch._lazy_clone(base)                                         # shares its memory until somebody writes
    _host_call(out)
    assert not torch._C._is_cow_tensor(out) and out.data_ptr() != base.data_ptr()


@pytest.mark.parametrize("stream", [0, np.int64(0)])
def test_a_stream_is_whatever_is_a_handle(stream):
    _host_call(torch.zeros(2, 4, 64, dtype=torch.bfloat16), stream)


def test_a_module_of_another_torch_is_neither_kept_nor_loaded(tmp_path, monkeypatch):
    build.build_library()
    assert build.binding_made_for() == build.binding_abi()
    stamp = tmp_path / "stamp"
    stamp.write_text(build.binding_abi().replace("torch ", "torch 1."))    # as a torch upgrade leaves it
    monkeypatch.setattr(build, "BINDING_FOR", str(stamp))
    commands = []
    monkeypatch.setattr(build, "_run", lambda cmd, verbose, what: commands.append(what))
    with pytest.raises(ImportError, match="stale"):
        kvattn._NativeLoader().kv_append
    build.build_library()
    assert commands == ["_kvattn_native.so"]                                  # rebuilt, and the library is not
    assert stamp.read_text() == build.binding_abi()
