"""The three ways the tensor-core extend kernel hands out its work (the plan's list, one item per cluster of CTAs, spans of
KV steps), at the sizes where each begins, against the oracle; and the entry points that share them, bit for bit."""
import numpy as np
import pytest
import torch

from paper_2607_23815_b200 import kvattn, synth
from harness import Batch, DualPool, assert_close, run_extend

pytestmark = pytest.mark.gpu


def _i32(x):
    return torch.tensor(np.asarray(x), dtype=torch.int32, device="cuda")


def _check(geom, P, E, seed, what):
    L = [p + e for p, e in zip(P, E)]
    dp = DualPool(geom, sum(synth.pages_needed(max(x, 1), 16) for x in L) + 2, seed=seed)
    b = Batch(dp, [max(x, 1) for x in L])
    b.write([(i, 0, L[i]) for i in range(len(L)) if L[i] > 0])
    res = run_extend(dp, b, P, E, impl=2)
    assert kvattn.kv_last_async_status(dp.pool) == kvattn.KV_OK
    assert_close(res, what)
    # the same call once more, through the plan entry points, and beside a decode set: the same bits
    hq, q, bt, ml = geom.n_q_heads, res["q"], torch.from_numpy(b.block_tables()).cuda(), max(L)
    cu, pl, el = _i32(np.concatenate([[0], np.cumsum(E)])), _i32(P), _i32(E)
    dec_rows = [i for i in range(len(L)) if L[i] > 0][:3]
    qd, ctx, btd = q[:len(dec_rows)].contiguous(), _i32([L[i] for i in dec_rows]), bt[dec_rows].contiguous()
    ws = torch.empty(kvattn.attn_workspace_bytes(dp.pool, hq, len(P), int(q.shape[0]), ml, len(dec_rows), ml), dtype=torch.uint8,
                     device="cuda")
    for how in ("plain", "planned", "mixed"):
        out, lse = torch.full_like(q, float("nan")), torch.full((q.shape[0], hq), float("nan"), device="cuda")
        if how == "plain":
            kvattn.attn_extend(dp.pool, q, cu, bt, pl, el, max(E), ml, geom.scale, out, lse, ws)
        elif how == "planned":
            kvattn.attn_extend_plan(dp.pool, hq, cu, bt, pl, el, int(q.shape[0]), max(E), ml, ws)
            kvattn.attn_extend_planned(dp.pool, q, cu, bt, pl, el, max(E), ml, geom.scale, out, lse, ws)
        else:
            od, ld = torch.empty_like(qd), torch.empty((len(dec_rows), hq), device="cuda")
            kvattn.attn_mixed(dp.pool, hq, geom.scale, kvattn.extend_args(q, cu, bt, pl, el, max(E), ml, out, lse),
                              kvattn.decode_args(qd, btd, ctx, ml, od, ld), ws)
        torch.cuda.synchronize()
        assert np.array_equal(synth.bf16_bits(out), res["o_bits"]), (what, how)
        assert np.array_equal(lse.cpu().numpy(), res["lse_raw"]), (what, how)
    # a workspace that holds no partial results still serves (another schedule, other roundings)
    small = torch.empty(1 << 20, dtype=torch.uint8, device="cuda")
    out, lse = torch.full_like(q, float("nan")), torch.full((q.shape[0], hq), float("nan"), device="cuda")
    kvattn.attn_extend(dp.pool, q, cu, bt, pl, el, max(E), ml, geom.scale, out, lse, small)
    torch.cuda.synchronize()
    res.update(o=out.float().cpu().numpy().astype(np.float64), lse=lse.cpu().numpy().astype(np.float64))
    assert_close(res, what + ", small workspace")
    assert kvattn.kv_last_async_status(dp.pool) == kvattn.KV_OK
    dp.close()


@pytest.mark.parametrize("hq,hkv,d", [(8, 2, 128), (8, 1, 64), (2, 2, 128)])
@pytest.mark.parametrize("total", [384, 385, 512, 640, 769, 1024, 1153, 4200])
def test_one_item_per_cluster_of_every_size(total, hq, hkv, d):
    # 3 KV steps (one CTA), then 4, 6 and 8 CTAs per item with one, two or more steps each; the longest takes the kernel
    # variant that does not search for the row maximum
    _check(synth.Geometry(hq, hkv, d), [total - 37], [37], 900 + total, f"cluster {total}")


def test_clusters_with_ragged_sequences():
    # sequences with fewer steps than CTAs, empty ones, tiles that see fewer keys than their partner, several tile pairs
    P = [1000, 0, 3, 0, 500, 120, 1023]
    E = [33, 200, 1, 0, 65, 16, 1]
    _check(synth.Geometry(8, 2, 128), P, E, 950, "ragged clusters")
    _check(synth.Geometry(16, 2, 64), P, E, 951, "ragged clusters, D 64")


@pytest.mark.parametrize("batch,long,hq,hkv,d", [(40, 3000, 8, 2, 128), (100, 4200, 8, 2, 64), (45, 4100, 4, 2, 128)])
def test_spans_cut_long_items(batch, long, hq, hkv, d):
    # few long items among many short ones: the long ones are cut into several spans, the short ones share one
    rng = np.random.default_rng(batch)
    P = [int(x) for x in rng.integers(0, 300, size=batch)]
    E = [int(x) for x in rng.integers(0, 60, size=batch)]
    P[0], E[0], P[batch // 2], E[batch // 2], P[-1], E[-1] = long - 50, 50, long - 61, 61, long // 2, 64
    _check(synth.Geometry(hq, hkv, d), P, E, 960 + batch, f"spans {batch}")


@pytest.mark.parametrize("long,batch", [(1500, 3), (3000, 40)])
def test_append_and_extend_right_behind_what_writes_their_inputs(long, batch):
    # clusters and spans read lengths, tables and Q while the call's own append runs: everything queued before that is final.
    # Each step's query, keys, lengths and table come from the kernels just in front of it; with and without waiting between.
    hq, hkv, d, e, steps = 8, 2, 128, 24, 4
    rng = np.random.default_rng(batch)
    P = [long] + [int(x) for x in rng.integers(0, 200, size=batch - 1)]
    need = [-(-(p + e * steps) // 16) for p in P]
    width, total = max(need), sum(need)
    table = np.full((batch, width), -1, dtype=np.int32)
    ids = rng.permutation(total).astype(np.int32)
    for i, k in enumerate(need):
        table[i, :k], ids = ids[:k], ids[k:]
    pages = [torch.zeros((total, hkv, 16, d), dtype=torch.bfloat16, device="cuda") for _ in range(2)]
    pool = kvattn.kv_pool_create_ex(total, 16, hkv, d, *pages)
    ids_all = kvattn.kv_alloc(pool, total)
    assert sorted(ids_all) == list(range(total))
    gen = torch.Generator(device="cuda").manual_seed(batch)
    randn = lambda *s: torch.randn(s, generator=gen, device="cuda", dtype=torch.bfloat16)
    k0, v0, q0 = randn(sum(P), hkv, d), randn(sum(P), hkv, d), randn(batch * e, hq, d)
    cu_p, cu = _i32(np.concatenate([[0], np.cumsum(P)])), _i32(np.arange(batch + 1) * e)
    bt_all, el, scale, ml = _i32(table), _i32([e] * batch), float(np.float32(d ** -0.5)), max(P) + e * steps
    ws = torch.empty(kvattn.attn_workspace_bytes(pool, hq, batch, batch * e, ml, 0, 0), dtype=torch.uint8, device="cuda")
    runs = []
    for wait in (True, False, False):
        for t in pages:
            t.zero_()
        kvattn.kv_append(pool, k0, v0, cu_p, _i32([0] * batch), None, bt_all)
        q, pl, bt, outs = q0.clone(), _i32(P), torch.full_like(bt_all, -1), []
        out, lse = torch.empty_like(q), torch.empty((batch * e, hq), device="cuda")
        for _ in range(steps):
            bt.copy_(bt_all)                       # (the table of the step is written in front of the call)
            kn, vn = q[:, :hkv].contiguous(), q[:, hkv:2 * hkv].contiguous()
            if wait:
                torch.cuda.synchronize()
            kvattn.attn_extend_append(pool, q, kn, vn, cu, bt, pl, el, e, ml, scale, out, lse, ws)
            if wait:
                torch.cuda.synchronize()
            outs.append((out.clone(), lse.clone()))
            pl += el
            q = (out * 4).contiguous()
            bt.fill_(-1)
        torch.cuda.synchronize()
        runs.append(outs)
    assert kvattn.kv_last_async_status(pool) == kvattn.KV_OK
    for other in runs[1:]:
        for (o1, l1), (o2, l2) in zip(runs[0], other):
            assert torch.equal(o1.view(torch.int16), o2.view(torch.int16)) and torch.equal(l1, l2)
    kvattn.kv_pool_destroy(pool)
