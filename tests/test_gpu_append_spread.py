"""Appends at the sizes where their blocks are spread differently over the SMs: the pages hold exactly the rows, the slots behind a
segment's last token are cleared, and the call that appends and extends stores and computes the same."""
import numpy as np
import pytest
import torch

from paper_2607_23815_b200 import kvattn, synth
from harness import Batch, DualPool, assert_close, extend_schedule, run_extend

pytestmark = pytest.mark.gpu
SMS = torch.cuda.get_device_properties(0).multi_processor_count if torch.cuda.is_available() else 148


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


@pytest.mark.parametrize("total", [d + e * SMS for e in (1, 8, 16, 24) for d in (0, 1)])
def test_rows_of_more_than_128_chunks(total):
    test_rows_and_cleared_tails(total, 32, 128)


@pytest.mark.parametrize("geom,lens,how", [((8, 8, 128), [SMS] * 16, "clusters"),              # two blocks to an SM, full
                                           ((8, 8, 128), [SMS] * 16 + [1], "clusters"),        # three
                                           ((8, 8, 128), [SMS] * 18 + [6 * SMS], "spans"),     # three, full
                                           ((8, 8, 128), [SMS] * 18 + [6 * SMS + 1], "spans"),  # not spread
                                           ((16, 16, 128), [SMS] * 8, "clusters"), ((16, 16, 128), [SMS] * 7 + [SMS + 1], "clusters"),
                                           ((16, 4, 64), [40] * 30, "clusters"), ((8, 1, 128), [64, 80] * 9, "clusters")])
def test_in_front_of_attention_without_a_plan(geom, lens, how):
    # the append of the call itself, at the edges of its rules, in front of clusters and spans: the pages, O and LSE of two calls, and the oracle's
    geom, n, total = synth.Geometry(*geom), len(lens), sum(lens)
    P = [200 + 7 * (i % 5) for i in range(n)] if how == "clusters" else [40 * (i % 3) for i in range(n - 1)] + [2500]
    L = [p + e for p, e in zip(P, lens)]
    dp = DualPool(geom, sum(synth.pages_needed(x, 16) for x in L) + 2, seed=total)
    b = Batch(dp, L)
    b.write([(i, 0, P[i]) for i in range(n) if P[i]])
    k, v = (torch.cat(x) for x in zip(*[b.kv(i, P[i], L[i]) for i in range(n)]))
    q = torch.cat([b.q(i, P[i], L[i]) for i in range(n)]).contiguous()
    cu, bt, pl, el = _i32(np.concatenate([[0], np.cumsum(lens)])), torch.from_numpy(b.block_tables()).cuda(), _i32(P), _i32(lens)
    ws = torch.empty(kvattn.attn_workspace_bytes(dp.pool, geom.n_q_heads, n, total, max(L), 0, 0), dtype=torch.uint8, device="cuda")
    assert extend_schedule(dp.pool, geom.n_q_heads, q, cu, bt, pl, el, max(lens), max(L), geom.scale, ws) == how
    out, lse = torch.full_like(q, float("nan")), torch.full((total, geom.n_q_heads), float("nan"), device="cuda")
    kvattn.attn_extend_append(dp.pool, q, k, v, cu, bt, pl, el, max(lens), max(L), geom.scale, out, lse, ws)
    for i in range(n):
        at = int(np.sum(lens[:i]))
        dp.host.append(b.rows[i], P[i], synth.bf16_bits(k[at:at + lens[i]]), synth.bf16_bits(v[at:at + lens[i]]))
    res = run_extend(dp, b, P, lens)                                # attn_extend over the pages that the call has stored, and the oracle
    assert_close(res, f"{how}, {total} tokens")
    assert np.array_equal(synth.bf16_bits(out), res["o_bits"]) and np.array_equal(lse.cpu().numpy(), res["lse_raw"])
    assert kvattn.kv_last_async_status(dp.pool) == kvattn.KV_OK
    dp.close()
