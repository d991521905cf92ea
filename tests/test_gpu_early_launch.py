"""Library calls right behind one another, no other kernel between them: each is resident while the one in front still stores
what it will read.  The same bits as with a wait after every call."""
import numpy as np
import pytest
import torch

from paper_2607_23815_b200 import kvattn, synth
from harness import Batch, DualPool

pytestmark = pytest.mark.gpu


def _i32(x):
    return torch.tensor(np.asarray(x), dtype=torch.int32, device="cuda")


def _runs(body, times=4):
    ref = body(torch.cuda.synchronize)
    torch.cuda.synchronize()
    for _ in range(times):
        got = body(lambda: None)
        torch.cuda.synchronize()
        for (o1, l1), (o2, l2) in zip(ref, got):
            assert torch.equal(o1.view(torch.int16), o2.view(torch.int16)) and torch.equal(l1, l2)
    return ref


@pytest.mark.parametrize("impl", [1, 2])
@pytest.mark.parametrize("lens,hq,hkv,d", [([40], 8, 2, 128), ([90, 33, 64], 32, 8, 64), ([700, 16] + [150] * 60, 32, 8, 128), ([60] * 160, 16, 8, 64)])
def test_decode_behind_the_append_that_rewrites_its_pages(impl, lens, hq, hkv, d):
    # two sets of keys and values are stored in turn over the same pages, and a decode call follows each
    geom, steps = synth.Geometry(hq, hkv, d), 6
    dp = DualPool(geom, sum(synth.pages_needed(n, 16) for n in lens) + 2, seed=sum(lens) % 97, with_oracle=False)
    b = Batch(dp, lens)
    gen = torch.Generator(device="cuda").manual_seed(1)
    randn = lambda *s: torch.randn(s, generator=gen, device="cuda", dtype=torch.bfloat16)
    sets = [(randn(sum(lens), hkv, d), randn(sum(lens), hkv, d)) for _ in range(2)]
    q, cu, zero = randn(len(lens), hq, d), _i32(np.concatenate([[0], np.cumsum(lens)])), _i32([0] * len(lens))
    bt, ctx = torch.from_numpy(b.block_tables()).cuda(), _i32(lens)

    def body(wait):
        outs = [(torch.full_like(q, 7.0), torch.full((len(lens), hq), 7.0, device="cuda")) for _ in range(steps)]
        torch.cuda.synchronize()
        for s, (o, l) in enumerate(outs):
            kvattn.kv_append(dp.pool, *sets[s % 2], cu, zero, None, bt)
            wait()
            kvattn.attn_decode(dp.pool, q, bt, ctx, max(lens), geom.scale, o, l, None)
            wait()
        return outs

    kvattn.kvattn_set_decode_impl(impl)
    try:
        ref = _runs(body)
    finally:
        kvattn.kvattn_set_decode_impl(0)
    assert torch.equal(ref[0][0], ref[2][0]) and not torch.equal(ref[0][0], ref[1][0])
    assert kvattn.kv_last_async_status(dp.pool) == kvattn.KV_OK
    dp.close()


@pytest.mark.parametrize("impl", [1, 2])
@pytest.mark.parametrize("ctx", [40, 900])
def test_two_buffers_in_turn(impl, ctx):
    # each call reads what the call in front stores and stores over what that one reads
    geom = synth.Geometry(8, 2, 128)
    dp = DualPool(geom, 128, seed=15, with_oracle=False)
    b = Batch(dp, [ctx, 33])
    b.write([(0, 0, ctx), (1, 0, 33)])
    bt, cl = torch.from_numpy(b.block_tables()).cuda(), _i32([ctx, 33])
    q0 = torch.cat([b.q(0, ctx - 1, ctx), b.q(1, 32, 33)]).contiguous()

    def body(wait):
        x, y, lse = q0.clone(), torch.full_like(q0, 7.0), torch.full((2, 8), 7.0, device="cuda")
        torch.cuda.synchronize()
        for _ in range(9):
            kvattn.attn_decode(dp.pool, x, bt, cl, ctx, geom.scale, y, lse, None)
            wait()
            x, y = y, x
        return [(x, lse), (y, lse)]

    kvattn.kvattn_set_decode_impl(impl)
    try:
        _runs(body, times=10)
    finally:
        kvattn.kvattn_set_decode_impl(0)
    dp.close()


@pytest.mark.parametrize("P,E", [([1400], [30]), ([700, 0, 90], [20, 150, 1]), ([300] * 60, [70] * 60)])
def test_extend_behind_the_append_that_rewrites_its_prefix(P, E):
    geom, steps = synth.Geometry(8, 2, 128), 6
    L = [p + e for p, e in zip(P, E)]
    dp = DualPool(geom, sum(synth.pages_needed(n, 16) for n in L) + 2, seed=16, with_oracle=False)
    b = Batch(dp, L)
    gen = torch.Generator(device="cuda").manual_seed(2)
    randn = lambda *s: torch.randn(s, generator=gen, device="cuda", dtype=torch.bfloat16)
    sets = [(randn(sum(L), 2, 128), randn(sum(L), 2, 128)) for _ in range(2)]
    q, cu_l, zero = randn(sum(E), 8, 128), _i32(np.concatenate([[0], np.cumsum(L)])), _i32([0] * len(L))
    bt, cu, pl, el = torch.from_numpy(b.block_tables()).cuda(), _i32(np.concatenate([[0], np.cumsum(E)])), _i32(P), _i32(E)
    ws = torch.empty(kvattn.attn_workspace_bytes(dp.pool, 8, len(P), sum(E), max(L)), dtype=torch.uint8, device="cuda")

    def body(wait):
        outs = [(torch.full_like(q, 7.0), torch.full((sum(E), 8), 7.0, device="cuda")) for _ in range(steps)]
        torch.cuda.synchronize()
        for s, (o, l) in enumerate(outs):
            kvattn.kv_append(dp.pool, *sets[s % 2], cu_l, zero, None, bt)
            wait()
            kvattn.attn_extend(dp.pool, q, cu, bt, pl, el, max(E), max(L), geom.scale, o, l, ws)
            wait()
        return outs

    ref = _runs(body)
    assert torch.equal(ref[0][0], ref[2][0]) and not torch.equal(ref[0][0], ref[1][0])
    assert kvattn.kv_last_async_status(dp.pool) == kvattn.KV_OK
    dp.close()
