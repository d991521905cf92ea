"""Kernels that are launched early are resident while the kernels in front of them still write: none of their code may load
through the read-only path, which is for data that nobody writes during a kernel's life (no GPU needed)."""
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2607_23815_b200", "csrc")


def _code(name):
    text = open(os.path.join(CSRC, name)).read()
    return re.sub(r"//[^\n]*", "", re.sub(r"/\*.*?\*/", "", text, flags=re.S))


def _kernels(text):
    """The file's kernels by name: from __global__ to the closing brace at the start of a line."""
    return {m.group(1): m.group(0) for m in re.finditer(r"__global__ void (?:__launch_bounds__\([^)]*\)\s*)?(\w+)\(.*?^\}", text, flags=re.S | re.M)}


FILES = sorted(f for f in os.listdir(CSRC) if f.endswith((".cu", ".cuh")))
EARLY = {f: [n for n, body in _kernels(_code(f)).items() if "dependency_wait()" in body] for f in FILES}


def test_the_kernels_that_wait_are_found():
    found = {n for names in EARLY.values() for n in names}
    assert {"append_kernel", "attn_decode_kernel", "attn_extend_tc_kernel", "extend_prologue_kernel", "append_prologue_kernel",
            "extend_tc_plan_kernel", "span_combine_kernel"} <= found


@pytest.mark.parametrize("name", [f for f in FILES if EARLY[f]] + ["append.cuh", "page_mma.cuh"])
def test_no_read_only_loads_in_early_kernels(name):
    text = _code(name)
    if name == "pool.cu":                       # (holds kernels with an ordinary launch as well)
        text = "".join(body for n, body in _kernels(text).items() if n in EARLY[name])
    assert not re.search(r"__ldg\s*\(|\.nc\b", text), f"{name}: read-only load in code of a kernel that is launched early"


def test_blocks_of_the_next_kernel_are_not_let_in_to_wait():
    # kv_append: not before its own blocks have waited; decode: not before a warp has read its pages (attn_mixed's extend kernel lets
    # the decode kernel in at once, which runs beside it)
    append, decode = (_kernels(_code(f))[k] for f, k in (("pool.cu", "append_kernel"), ("attn_decode.cu", "attn_decode_kernel")))
    assert "launch_dependents" not in append and append.index("dependency_wait") < append.index("append_tokens<kMaxPerLane, true>")
    assert decode.index("launch_dependents") > decode.rindex("page_step")
    store = _code("append.cuh")
    assert store.index("block_tables + ") < store.index("launch_dependents") < store.index("= kk[i]")
