"""Appends at the sizes where their blocks are spread differently over the SMs: the pages hold exactly the rows, the slots behind a
segment's last token are cleared, and the call that appends and extends stores and computes the same."""
import numpy as np
import pytest
import torch

from paper_2607_23815_b200 import kvattn

pytestmark = pytest.mark.gpu


def _i32(x):
    return torch.tensor(np.asarray(x), dtype=torch.int32, device="cuda")


def _totals():
    sms = torch.cuda.get_device_properties(0).multi_processor_count if torch.cuda.is_available() else 148
    edges = (sms - 1, sms, 2 * sms, 8 * sms, 16 * sms, 24 * sms)
    return sorted({1, 2, 37} | {e + d for e in edges for d in (0, 1)} | {32 * (sms - 1) + 1})


@pytest.mark.parametrize("hkv,d", [(2, 64), (8, 128)])
@pytest.mark.parametrize("total", _totals())
def test_rows_and_cleared_tails(total, hkv, d):
    rng = np.random.default_rng(total)
    lens = []                                              # segments of one token (decodes) and of up to 200, some empty
    while sum(lens) < total:
        lens.append(min(total - sum(lens), int(rng.choice([0, 1, 1, 17, 64, 200]))))
    start = [int(x) for x in rng.integers(0, 40, size=len(lens))]
    need = [max(1, -(-(s + n) // 16)) for s, n in zip(start, lens)]
    table, ids = np.full((len(lens), max(need)), -1, dtype=np.int32), rng.permutation(sum(need)).astype(np.int32)
    for i, k in enumerate(need):
        table[i, :k], ids = ids[:k], ids[k:]
    gen = torch.Generator(device="cuda").manual_seed(total)
    k, v = (torch.randn((total, hkv, d), generator=gen, device="cuda", dtype=torch.bfloat16) for _ in range(2))
    bt, cu, hq, e_max, ml = _i32(table), _i32(np.concatenate([[0], np.cumsum(lens)])), 4 * hkv, max(max(lens), 1), 16 * max(need)
    q = torch.randn((total, hq, d), generator=gen, device="cuda", dtype=torch.bfloat16)
    images = []
    for fused in (False, True):
        pages = [torch.full((sum(need), hkv, 16, d), 3.0, dtype=torch.bfloat16, device="cuda") for _ in range(2)]
        pool = kvattn.kv_pool_create_ex(sum(need), 16, hkv, d, *pages)
        out, lse = torch.empty_like(q), torch.empty((total, hq), device="cuda")
        ws = torch.empty(kvattn.attn_workspace_bytes(pool, hq, len(lens), total, ml, 0, 0), dtype=torch.uint8, device="cuda")
        args = (cu, bt, _i32(start), _i32(lens), e_max, ml, d ** -0.5, out, lse, ws)
        if fused:
            kvattn.attn_extend_append(pool, q, k, v, *args)
        else:
            kvattn.kv_append(pool, k, v, cu, _i32(start), None, bt)
            kvattn.attn_extend(pool, q, *args)
        torch.cuda.synchronize()
        assert kvattn.kv_last_async_status(pool) == kvattn.KV_OK
        images.append((pages, out, lse))
        if not fused:
            at = 0
            for i, n in enumerate(lens):
                if n == 0:
                    continue
                whole = (start[i] + n + 15) // 16 * 16
                got = [torch.empty((whole, hkv, d), dtype=torch.bfloat16, device="cuda") for _ in range(2)]
                kvattn.kv_gather(pool, bt[i].contiguous(), whole, *got)
                for g, rows in zip(got, (k, v)):
                    assert torch.equal(g[start[i]:start[i] + n].view(torch.int16), rows[at:at + n].view(torch.int16)), i
                    assert not g[start[i] + n:].view(torch.int16).any(), i
                    assert bool((g[:start[i]] == 3.0).all()), i
                at += n
        kvattn.kv_pool_destroy(pool)
    (p0, o0, l0), (p1, o1, l1) = images
    assert all(torch.equal(a.view(torch.int16), b.view(torch.int16)) for a, b in zip(p0, p1))
    assert torch.equal(o0.view(torch.int16), o1.view(torch.int16)) and torch.equal(l0, l1)
