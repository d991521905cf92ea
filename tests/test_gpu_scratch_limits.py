"""The smallest workspaces that the calls take: the size of the extend kernel's work list and nothing for partial results."""
import numpy as np
import pytest
import torch

from paper_2607_23815_b200 import kvattn, synth
from harness import Batch, DualPool

pytestmark = pytest.mark.gpu


def _i32(x):
    return torch.tensor(np.asarray(x), dtype=torch.int32, device="cuda")


def _up(x):
    return (x + 255) // 256 * 256


def _list_bytes(batch, total_q):                 # 256 bytes of counters, then a 32-byte record per possible item
    return 256 + _up(32 * (total_q * 8 // 256 + batch + 1))


def _buffer(n, shift=0):
    """n bytes that start `shift` behind a 256-byte boundary, with a guard behind them."""
    whole = torch.full((n + shift + 4096,), 0xA5, dtype=torch.uint8, device="cuda")
    assert whole.data_ptr() % 256 == 0
    return whole[shift:shift + n], whole


def _same(a, b):                                 # another schedule, other roundings: two results within two bf16 roundings
    (o1, l1), (o2, l2) = a, b
    return bool(((o1.float() - o2.float()).abs() <= 8e-3 + 2.0 ** -5 * o2.float().abs()).all()) and bool(((l1 - l2).abs() <= 1e-4).all())


@pytest.mark.parametrize("P,E,hq,hkv,d", [([1500], [37], 8, 2, 128), ([300, 20, 700], [70, 5, 33], 8, 1, 64), ([40] * 60, [20] * 60, 16, 8, 128)])
def test_the_least_workspace(P, E, hq, hkv, d):
    geom, B, T = synth.Geometry(hq, hkv, d), len(P), sum(E)
    L = [p + e for p, e in zip(P, E)]
    dp = DualPool(geom, sum(synth.pages_needed(x, 16) for x in L) + 2, seed=91, with_oracle=False)
    b = Batch(dp, L)
    b.write([(i, 0, x) for i, x in enumerate(L)])
    q = torch.cat([b.q(i, P[i], L[i]) for i in range(B)]).contiguous()
    ks, vs = zip(*[b.kv(i, P[i], L[i]) for i in range(B)])
    k, v = torch.cat(ks).contiguous(), torch.cat(vs).contiguous()
    bt, cu, pl, el, ml = torch.from_numpy(b.block_tables()).cuda(), _i32(np.concatenate([[0], np.cumsum(E)])), _i32(P), _i32(E), max(L)
    qd, ctx = q[:B].contiguous(), _i32(L)
    dec_bytes = kvattn.attn_workspace_bytes(dp.pool, hq, 0, 0, 0, B, ml) - 256
    need = _list_bytes(B, T)

    def call(how, ws):
        out, lse = torch.full_like(q, float("nan")), torch.full((T, hq), float("nan"), device="cuda")
        args = (cu, bt, pl, el, max(E), ml, geom.scale, out, lse)
        if how == "extend":
            kvattn.attn_extend(dp.pool, q, *args, ws)
        elif how == "append":
            kvattn.attn_extend_append(dp.pool, q, k, v, *args, ws)
        elif how == "planned":
            kvattn.attn_extend_plan(dp.pool, hq, cu, bt, pl, el, T, max(E), ml, ws)
            kvattn.attn_extend_planned(dp.pool, q, *args, ws)
        elif how == "mixed":
            kvattn.attn_mixed(dp.pool, hq, geom.scale, kvattn.extend_args(q, cu, bt, pl, el, max(E), ml, out, lse),
                              kvattn.decode_args(qd, bt, ctx, ml, torch.empty_like(qd), torch.empty((B, hq), device="cuda")), ws)
        torch.cuda.synchronize()
        return out, lse

    full = torch.empty(kvattn.attn_workspace_bytes(dp.pool, hq, B, T, ml, B, ml), dtype=torch.uint8, device="cuda")
    want = call("extend", full)
    for how in ("extend", "append", "planned", "mixed"):
        n = need + dec_bytes if how == "mixed" else need
        for shift in (0, 16):                                       # (the list takes any 16-byte boundary)
            ws, whole = _buffer(n, shift)
            assert _same(call(how, ws), want), (how, shift)
            assert bool((whole[:shift] == 0xA5).all()) and bool((whole[shift + n:] == 0xA5).all()), (how, shift)
            with pytest.raises(kvattn.KvError) as e:
                call(how, ws[:n - 1])
            assert e.value.status == kvattn.KV_ERR_WORKSPACE, (how, shift)
    # the host step: its copies of the arrays, the list, 256 bytes
    host = [t.cpu() for t in (q, k, v, cu, bt, pl, el)]
    arrays = sum(_up(t.numel() * t.element_size()) for t in host) + _up(q.numel() * 2) + _up(T * hq * 4)
    n = arrays + _up(need) + 256
    out, lse = torch.zeros(q.shape, dtype=torch.bfloat16), torch.zeros((T, hq))
    staging, whole = _buffer(n)
    kvattn.attn_extend_host(dp.pool, *host, max(E), ml, geom.scale, out, lse, staging)
    torch.cuda.synchronize()
    assert _same((out.cuda(), lse.cuda()), want) and bool((whole[n:] == 0xA5).all())
    with pytest.raises(kvattn.KvError) as e:
        kvattn.attn_extend_host(dp.pool, *host, max(E), ml, geom.scale, out, lse, staging[:n - 1])
    assert e.value.status == kvattn.KV_ERR_WORKSPACE
    assert kvattn.kv_last_async_status(dp.pool) == kvattn.KV_OK
    dp.close()


@pytest.mark.parametrize("hq,hkv,d", [(8, 2, 128), (8, 1, 64)])
def test_the_least_workspace_of_a_fan_out(hq, hkv, d):
    geom, parents, n_child, children = synth.Geometry(hq, hkv, d), [640, 160], [3, 2], [20, 9, 33, 5, 17]
    dp = DualPool(geom, 128, seed=92, with_oracle=False)
    pb, cb = Batch(dp, parents), Batch(dp, children, uid0=100)
    pb.write([(i, 0, n) for i, n in enumerate(parents)])
    cb.write([(i, 0, n) for i, n in enumerate(children)])
    q = torch.cat([cb.q(i, 0, n) for i, n in enumerate(children)]).contiguous()
    cu, cc, T = np.concatenate([[0], np.cumsum(children)]), np.concatenate([[0], np.cumsum(n_child)]), sum(children)
    rows = [int(cu[cc[g + 1]] - cu[cc[g]]) for g in range(2)]

    def call(ws):
        out, lse = torch.full_like(q, float("nan")), torch.full((T, hq), float("nan"), device="cuda")
        kvattn.attn_extend_shared(dp.pool, q, _i32(cu), _i32(cc), torch.from_numpy(pb.block_tables()).cuda(), _i32(parents),
                                  torch.from_numpy(cb.block_tables()).cuda(), _i32(children), max(children), max(rows), max(parents),
                                  geom.scale, out, lse, ws)
        torch.cuda.synchronize()
        return out, lse

    full = kvattn.attn_extend_shared_workspace_bytes(dp.pool, hq, 2, 5, T, max(parents))
    want = call(torch.empty(full, dtype=torch.uint8, device="cuda"))
    n = _up(4 * (2 * 2 + 1 + 5)) + _up(T * hq * d * 2) + _up(T * hq * 4) + _up(_list_bytes(5, T)) + 256
    assert n < full
    ws, whole = _buffer(n)
    assert _same(call(ws), want) and bool((whole[n:] == 0xA5).all())
    with pytest.raises(kvattn.KvError) as e:
        call(ws[:n - 1])
    assert e.value.status == kvattn.KV_ERR_WORKSPACE
    dp.close()
