"""Keys that are not numbers: every row that sees one has no result, whichever way the work is split, and no other row changes.

A pool in poison mode overwrites evicted pages with NaN so that a table that still names one shows; that only works if no
merge of partial results leaves the broken part out."""
import numpy as np
import pytest
import torch

from paper_2607_23815_b200 import kvattn, synth
from harness import Batch, DualPool, extend_schedule

pytestmark = pytest.mark.gpu

NAN, INF = 0x7FC0, 0x7F80


def _i32(x):
    return torch.tensor(np.asarray(x), dtype=torch.int32, device="cuda")


def _set_key(dp, row, pos, head, bits):
    """Overwrites dim 0 of the key at position pos of a table row; returns the bits it held."""
    at = kvattn.kv_pool_elem_offset(dp.pool, row[pos // 16], head, pos % 16, 0)
    old = int(dp.k_buf[at].item())
    dp.k_buf[at] = bits
    torch.cuda.synchronize()
    return old


def _extend_calls(geom, P, E, seed):
    """A pool with the batch in it and the ways to call the extend kernel over it."""
    L = [p + e for p, e in zip(P, E)]
    dp = DualPool(geom, sum(synth.pages_needed(max(x, 1), 16) for x in L) + 2, seed=seed, with_oracle=False)
    b = Batch(dp, [max(x, 1) for x in L])
    b.write([(i, 0, x) for i, x in enumerate(L) if x > 0])
    hq, ml = geom.n_q_heads, max(L)
    q = torch.cat([b.q(i, P[i], L[i]) for i in range(len(P))]).contiguous()
    bt, cu, pl, el = torch.from_numpy(b.block_tables()).cuda(), _i32(np.concatenate([[0], np.cumsum(E)])), _i32(P), _i32(E)
    ks, vs = zip(*[b.kv(i, P[i], L[i]) for i in range(len(P))])
    k_new, v_new = torch.cat(ks).contiguous(), torch.cat(vs).contiguous()
    qd, ctx, btd = q[:1].contiguous(), _i32([L[-1]]), bt[-1:].contiguous()
    ws = torch.empty(kvattn.attn_workspace_bytes(dp.pool, hq, len(P), int(q.shape[0]), ml, 1, ml), dtype=torch.uint8, device="cuda")
    small = torch.empty(1 << 18, dtype=torch.uint8, device="cuda")

    def call(how):
        out, lse = torch.full_like(q, 7.0), torch.full((q.shape[0], hq), 7.0, device="cuda")
        args = (cu, bt, pl, el, max(E), ml, geom.scale, out, lse)
        if how == "plain":
            kvattn.attn_extend(dp.pool, q, *args, ws)
        elif how == "no room for partial results":
            kvattn.attn_extend(dp.pool, q, *args, small)
        elif how == "planned":
            kvattn.attn_extend_plan(dp.pool, hq, cu, bt, pl, el, int(q.shape[0]), max(E), ml, ws)
            kvattn.attn_extend_planned(dp.pool, q, *args, ws)
        elif how == "append":                                     # (writes the suffix keys again: they are what they were)
            kvattn.attn_extend_append(dp.pool, q, k_new, v_new, *args, ws)
        else:
            od, ld = torch.empty_like(qd), torch.empty((1, hq), device="cuda")
            kvattn.attn_mixed(dp.pool, hq, geom.scale, kvattn.extend_args(q, cu, bt, pl, el, max(E), ml, out, lse),
                              kvattn.decode_args(qd, btd, ctx, ml, od, ld), ws)
        torch.cuda.synchronize()
        return out, lse

    schedule = extend_schedule(dp.pool, hq, q, cu, bt, pl, el, max(E), ml, geom.scale, ws)
    return dp, b, q, call, schedule


@pytest.mark.parametrize("schedule,P,E,hq,hkv,d", [
    ("clusters", [1116], [37], 8, 2, 128), ("clusters", [4163], [37], 8, 1, 64), ("clusters", [1500, 300], [70, 9], 8, 2, 64),
    ("spans", [2950] + [40] * 18 + [2939] + [130] * 20, [50] + [20] * 18 + [61] + [33] * 20, 8, 2, 128),
    ("spans", [4150] + [40] * 49 + [4139] + [130] * 49, [50] + [20] * 49 + [61] + [33] * 49, 8, 2, 64)])
def test_a_broken_key_reaches_every_row_that_sees_it(schedule, P, E, hq, hkv, d):
    geom = synth.Geometry(hq, hkv, d)
    dp, b, q, call, got_schedule = _extend_calls(geom, P, E, seed=41 + len(P))
    assert got_schedule == schedule
    G, cu = hq // hkv, np.concatenate([[0], np.cumsum(E)])
    ways = ("plain", "planned", "append", "mixed", "no room for partial results")
    clean = {how: call(how) for how in ways}
    broken = 0 if len(P) < 3 else len(P) // 2 - 1 if P[len(P) // 2 - 1] > 1000 else int(np.argmax(P))
    head = hkv - 1
    qv = q[cu[broken]:cu[broken + 1], head * G:(head + 1) * G, 0].float()
    for pos in (3, P[broken] // 2, P[broken] - 1, P[broken] + 5):    # the first, a middle and the last part of the keys
        for bits in (NAN, INF):
            for how in ways:
                old = _set_key(dp, b.rows[broken], pos, head, bits)
                if how == "append" and pos >= P[broken]:
                    _set_key(dp, b.rows[broken], pos, head, old)  # (the call would store the sound key over it)
                    continue
                out, lse = call(how)
                _set_key(dp, b.rows[broken], pos, head, old)
                want = torch.zeros(lse.shape, dtype=torch.bool, device="cuda")
                sees = (torch.arange(E[broken], device="cuda") + P[broken] >= pos)[:, None]
                # (an infinite key gives a score of -inf where the query's element is negative: no weight, a sound result)
                want[cu[broken]:cu[broken + 1], head * G:(head + 1) * G] = sees & (qv > 0) if bits == INF else sees.expand(-1, G)
                what = (schedule, how, pos, hex(bits))
                assert torch.equal(torch.isnan(out.float()).all(-1), want) and torch.equal(torch.isnan(out.float()).any(-1), want), what
                assert torch.equal(torch.isnan(lse), want), what
                if bits == NAN:                                    # rows that do not see the key keep their bits
                    assert torch.equal(out[~want], clean[how][0][~want]) and torch.equal(lse[~want], clean[how][1][~want]), what
    assert kvattn.kv_last_async_status(dp.pool) == kvattn.KV_OK
    dp.close()


@pytest.mark.parametrize("hq,hkv,d", [(8, 2, 128), (8, 1, 64)])
def test_a_broken_key_of_a_parent_reaches_its_children_only(hq, hkv, d):
    geom = synth.Geometry(hq, hkv, d)
    parents, n_child, children = [1200, 640], [3, 2], [20, 9, 33, 5, 17]
    dp = DualPool(geom, 256, seed=43, with_oracle=False)
    pb, cb = Batch(dp, parents), Batch(dp, children, uid0=100)
    pb.write([(i, 0, n) for i, n in enumerate(parents)])
    cb.write([(i, 0, n) for i, n in enumerate(children)])
    q = torch.cat([cb.q(i, 0, n) for i, n in enumerate(children)]).contiguous()
    cu, cc = np.concatenate([[0], np.cumsum(children)]), np.concatenate([[0], np.cumsum(n_child)])
    rows = [int(cu[cc[g + 1]] - cu[cc[g]]) for g in range(2)]
    ws = torch.empty(kvattn.attn_extend_shared_workspace_bytes(dp.pool, hq, 2, 5, int(q.shape[0]), max(parents)), dtype=torch.uint8, device="cuda")

    def call():
        out, lse = torch.full_like(q, 7.0), torch.full((q.shape[0], hq), 7.0, device="cuda")
        kvattn.attn_extend_shared(dp.pool, q, _i32(cu), _i32(cc), torch.from_numpy(pb.block_tables()).cuda(), _i32(parents),
                                  torch.from_numpy(cb.block_tables()).cuda(), _i32(children), max(children), max(rows), max(parents),
                                  geom.scale, out, lse, ws)
        torch.cuda.synchronize()
        return out, lse

    clean, G = call(), hq // hkv
    for pos in (0, 600, 1199):
        old = _set_key(dp, pb.rows[0], pos, 0, NAN)
        out, lse = call()
        _set_key(dp, pb.rows[0], pos, 0, old)
        want = torch.zeros(lse.shape, dtype=torch.bool, device="cuda")
        want[:rows[0], :G] = True
        assert torch.equal(torch.isnan(lse), want) and torch.equal(torch.isnan(out.float()).all(-1), want), pos
        assert torch.equal(out[~want], clean[0][~want]) and torch.equal(lse[~want], clean[1][~want]), pos
    dp.close()


@pytest.mark.parametrize("hq,hkv,d,lens", [(8, 2, 128, [4000, 70]), (8, 1, 64, [517]), (32, 8, 128, [90] * 80)])
def test_a_broken_key_reaches_its_decode_rows(hq, hkv, d, lens):
    geom = synth.Geometry(hq, hkv, d)                              # clusters of CTAs, and several pairs per CTA
    dp = DualPool(geom, sum(synth.pages_needed(n, 16) for n in lens) + 2, seed=44, with_oracle=False)
    b = Batch(dp, lens)
    b.write([(i, 0, n) for i, n in enumerate(lens)])
    q, bt, ctx = torch.cat([b.q(i, n - 1, n) for i, n in enumerate(lens)]).contiguous(), torch.from_numpy(b.block_tables()).cuda(), _i32(lens)
    ws = torch.empty(max(256, kvattn.attn_workspace_bytes(dp.pool, hq, 0, 0, 0, len(lens), max(lens))), dtype=torch.uint8, device="cuda")
    for pos in (0, lens[0] // 2, lens[0] - 1):
        old = _set_key(dp, b.rows[0], pos, 0, NAN)
        out, lse = torch.full_like(q, 7.0), torch.empty((len(lens), hq), device="cuda")
        kvattn.attn_decode(dp.pool, q, bt, ctx, max(lens), geom.scale, out, lse, ws)
        torch.cuda.synchronize()
        _set_key(dp, b.rows[0], pos, 0, old)
        want = torch.zeros(lse.shape, dtype=torch.bool, device="cuda")
        want[0, :hq // hkv] = True
        assert torch.equal(torch.isnan(out.float()).all(-1), want) and torch.equal(torch.isnan(out.float()).any(-1), want), pos
    dp.close()
