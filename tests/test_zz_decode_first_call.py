"""One decode call per device is enough before stream captures and frozen allocators: later calls of any shape, which may be the
first use of another variant of the kernel, neither load code nor change the free device memory.

Runs in a process of its own, where nothing has been loaded yet."""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

_SCRIPT = """
import time
import torch
from paper_2607_23815_b200 import kvattn
torch.cuda.init()
def state(d, hq, hkv, batch, ctx):
    pages = [torch.zeros((256, hkv, 16, d), dtype=torch.bfloat16, device="cuda") for _ in range(2)]
    pool = kvattn.kv_pool_create_ex(256, 16, hkv, d, *pages)
    n = -(-ctx // 16)
    bt = (torch.arange(batch * n, dtype=torch.int32, device="cuda") % 256).view(batch, n)
    return dict(pool=pool, pages=pages, bt=bt, cl=torch.full((batch,), ctx, dtype=torch.int32, device="cuda"), ctx=ctx,
                q=torch.ones((batch, hq, d), dtype=torch.bfloat16, device="cuda"), out=torch.empty((batch, hq, d), dtype=torch.bfloat16, device="cuda"),
                lse=torch.empty((batch, hq), device="cuda"))
# registers, ring, several pairs per CTA with either, at both head sizes
shapes = [(d, hq, hkv, batch, ctx) for d in (128, 64) for hq, hkv, batch, ctx in
          ((8, 2, 1, 40), (8, 2, 40, 1000), (32, 8, 300, 20), (32, 8, 300, 120), (8, 8, 300, 400))]
states = [state(*s) for s in shapes]
torch.cuda.synchronize()
side = torch.cuda.Stream()
def call(s, stream=None):
    kvattn.attn_decode_static(s["pool"], s["q"], s["bt"], s["cl"], s["ctx"], 0.125, s["out"], s["lse"], stream)
for _ in range(3):                                                # (the contract asks for one call; the clock wants a warm thread)
    call(states[0])
    torch.cuda.synchronize()
free, grew, late = torch.cuda.mem_get_info()[0], [], []
for s in states:
    if CAPTURE:
        g = torch.cuda.CUDAGraph()
        with torch.cuda.stream(side):
            g.capture_begin()
            call(s)
            g.capture_end()
        g.replay()
    else:
        times = []
        for _ in range(4):
            t0 = time.perf_counter()
            call(s)
            times.append(time.perf_counter() - t0)
            torch.cuda.synchronize()
        if times[0] > min(times[1:]) + 20e-6:                     # loading a variant takes 30 us and more
            late.append((times[0], min(times[1:])))
    torch.cuda.synchronize()
    grew.append(free - torch.cuda.mem_get_info()[0])
for s in states:
    assert float(s["out"].float().abs().max()) == 0.0 and kvattn.kv_last_async_status(s["pool"]) == 0   # (the values are zeros)
print("grew by", grew)
assert CAPTURE or not any(grew)                                   # (a graph has memory of its own)
assert len(late) <= 2, late                                       # (four variants are new; two for whatever else the host was doing)
print("done")
"""


@pytest.mark.parametrize("capture", [False, True])
def test_one_call_prepares_every_variant(capture):
    env = dict(os.environ, CUDA_MODULE_LOADING="LAZY")
    r = subprocess.run([sys.executable, "-c", _SCRIPT.replace("CAPTURE", str(capture))], capture_output=True, text=True, cwd=ROOT, timeout=600, env=env)
    assert r.returncode == 0 and "done" in r.stdout, (r.stdout, r.stderr[-3000:])
