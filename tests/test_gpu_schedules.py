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
