"""attn_extend_host from pinned and pageable buffers, in steps small enough for its copy kernel and larger ones, with
addresses that are not 16-byte aligned, one staging area and two in turn: the bits of the call on device tensors."""
import numpy as np
import pytest
import torch

from paper_2607_23815_b200 import kvattn, synth
from harness import Batch, DualPool

pytestmark = pytest.mark.gpu


def _host(t, pinned, shift=0):
    """A host copy of t; shift: elements by which it starts off its buffer's beginning."""
    flat = torch.empty(t.numel() + shift, dtype=t.dtype, pin_memory=pinned)
    view = flat[shift:shift + t.numel()].view(t.shape)
    view.copy_(t)
    return view


@pytest.mark.parametrize("pinned", [True, False, "mixed"])
@pytest.mark.parametrize("extend", [[5, 1], [60, 33], [600, 300, 1]])
def test_host_step_gives_the_bits_of_the_device_call(extend, pinned):
    geom = synth.Geometry(8, 2, 128)                       # the largest suffix set: 4.6 MB of rows, above the kernel's limit
    P = [37, 250, 16][:len(extend)]
    L = [p + e for p, e in zip(P, extend)]
    outs = []
    for way in ("device", "host"):
        dp = DualPool(geom, 256, seed=71, with_oracle=False)
        b = Batch(dp, L)
        b.write([(i, 0, P[i]) for i in range(len(P))])
        ks, vs = zip(*[b.kv(i, P[i], L[i]) for i in range(len(P))])
        k, v = torch.cat(ks).contiguous(), torch.cat(vs).contiguous()
        q = torch.cat([b.q(i, P[i], L[i]) for i in range(len(P))]).contiguous()
        i32 = lambda x: torch.tensor(np.asarray(x), dtype=torch.int32)
        cu, bt, pl, el = i32(np.concatenate([[0], np.cumsum(extend)])), torch.from_numpy(b.block_tables()), i32(P), i32(extend)
        bounds = (max(extend), max(L), geom.scale)
        if way == "device":
            out, lse = torch.empty_like(q), torch.empty((q.shape[0], 8), device="cuda")
            ws = torch.empty(kvattn.attn_workspace_bytes(dp.pool, 8, len(P), int(q.shape[0]), max(L)), dtype=torch.uint8, device="cuda")
            kvattn.attn_extend_append(dp.pool, q, k, v, cu.cuda(), bt.cuda(), pl.cuda(), el.cuda(), *bounds, out, lse, ws)
            outs.append((synth.bf16_bits(out), lse.cpu().numpy(), dp.device_image()))
        else:
            pin = lambda i: pinned if pinned != "mixed" else i % 2 == 0
            h = [_host(t, pin(i), shift=1 if t.dtype == torch.int32 else 0) for i, t in enumerate((q, k, v, cu, bt, pl, el))]
            size = kvattn.attn_extend_host_staging_bytes(dp.pool, 8, len(P), int(q.shape[0]), bt.shape[1], max(L))
            areas = [torch.empty(size, dtype=torch.uint8, device="cuda") for _ in range(2)]
            for step in range(5):                           # (an append of the same rows again changes nothing)
                o = _host(torch.full(q.shape, float("nan"), dtype=torch.bfloat16), pin(0))
                l = _host(torch.full((q.shape[0], 8), float("nan")), pin(1), shift=1)
                kvattn.attn_extend_host(dp.pool, *h, *bounds, o, l, areas[step % 2])
                torch.cuda.current_stream().synchronize()
                outs.append((synth.bf16_bits(o), l.numpy().copy(), dp.device_image()))
        assert kvattn.kv_last_async_status(dp.pool) == kvattn.KV_OK
        dp.close()
    for o in outs[1:]:
        assert np.array_equal(o[0], outs[0][0]) and np.array_equal(o[1], outs[0][1])
        assert np.array_equal(o[2][0], outs[0][2][0]) and np.array_equal(o[2][1], outs[0][2][1])


def _registered(t, region, at):
    """A host copy of t at byte `at` of a registered region."""
    view = region[at:at + t.numel() * t.element_size()].view(t.dtype).view(t.shape)
    view.copy_(t)
    return view


def test_buffers_inside_one_registration_are_copied_by_the_kernel():
    # memory that the caller registered instead of allocating it pinned; the last buffer ends with the region
    geom, P, E = synth.Geometry(8, 2, 128), [37, 250], [60, 33]
    L = [p + e for p, e in zip(P, E)]
    dp = DualPool(geom, 64, seed=72, with_oracle=False)
    b = Batch(dp, L)
    b.write([(i, 0, P[i]) for i in range(2)])
    ks, vs = zip(*[b.kv(i, P[i], L[i]) for i in range(2)])
    q = torch.cat([b.q(i, P[i], L[i]) for i in range(2)]).contiguous()
    i32 = lambda x: torch.tensor(np.asarray(x), dtype=torch.int32)
    arrays = [t.cpu() for t in (q, torch.cat(ks), torch.cat(vs), i32(np.concatenate([[0], np.cumsum(E)])), torch.from_numpy(b.block_tables()),
                                i32(P), i32(E), torch.zeros_like(q), torch.zeros((q.shape[0], 8)))]
    starts, at = [], 4
    for t in arrays:
        starts.append(at)
        at += t.numel() * t.element_size()
    outs, launches = [], []
    region = torch.zeros(at, dtype=torch.uint8)
    staging = torch.empty(kvattn.attn_extend_host_staging_bytes(dp.pool, 8, 2, int(q.shape[0]), arrays[4].shape[1], max(L)), dtype=torch.uint8,
                          device="cuda")
    for registered in (False, True):
        if registered:
            assert torch.cuda.cudart().cudaHostRegister(region.data_ptr(), at, 0) == torch.cuda.cudart().cudaError.success
        try:
            h = [_registered(t, region, s) for t, s in zip(arrays, starts)]
            before = kvattn.kvattn_launch_count()
            kvattn.attn_extend_host(dp.pool, *h[:7], max(E), max(L), geom.scale, h[7], h[8], staging)
            torch.cuda.synchronize()
            launches.append(kvattn.kvattn_launch_count() - before)
            outs.append((synth.bf16_bits(h[7]).copy(), h[8].numpy().copy()))
        finally:
            if registered:
                torch.cuda.synchronize()
                torch.cuda.cudart().cudaHostUnregister(region.data_ptr())
    assert launches[1] == launches[0] + 2                                  # one copy kernel in, one out
    assert np.array_equal(outs[0][0], outs[1][0]) and np.array_equal(outs[0][1], outs[1][1]) and np.any(outs[0][1] != 0)
    assert kvattn.kv_last_async_status(dp.pool) == kvattn.KV_OK
    dp.close()


@pytest.mark.parametrize("pinned", [True, False])
@pytest.mark.parametrize("areas", [1, 2, 5])
def test_steps_queued_behind_one_another_do_not_mix(areas, pinned):
    # every step has its own rows, lengths, tables and result buffers; nothing waits until all are queued.  Results below and
    # above what a kernel copies out (4 MB), rows below and above what it copies in (1 MB); more areas than the pool keeps track of
    geom = synth.Geometry(8, 2, 128)
    shapes = [([37, 250], [60, 33]), ([16, 5, 90], [400, 290, 10]), ([300], [1]), ([40, 17], [1300, 901]), ([129], [80]), ([64, 64], [1100, 1000]),
              ([700, 31], [20, 44]), ([3], [700])]
    need = [[synth.pages_needed(p + e, 16) for p, e in zip(P, E)] for P, E in shapes]
    i32 = lambda x: torch.tensor(np.asarray(x), dtype=torch.int32)
    outs = []
    for way in ("device", "host"):
        dp = DualPool(geom, sum(map(sum, need)) + 4, seed=73, with_oracle=False)
        batches = [Batch(dp, [p + e for p, e in zip(P, E)], uid0=100 * s) for s, (P, E) in enumerate(shapes)]
        steps = []
        for b, (P, E) in zip(batches, shapes):
            b.write([(i, 0, P[i]) for i in range(len(P))])
            ks, vs = zip(*[b.kv(i, P[i], P[i] + E[i]) for i in range(len(P))])
            q = torch.cat([b.q(i, P[i], P[i] + E[i]) for i in range(len(P))]).contiguous()
            arrays = (q, torch.cat(ks).contiguous(), torch.cat(vs).contiguous(), i32(np.concatenate([[0], np.cumsum(E)])),
                      torch.from_numpy(b.block_tables()), i32(P), i32(E))
            steps.append((arrays, (max(E), max(p + e for p, e in zip(P, E)), geom.scale)))
        if way == "device":
            for arrays, bounds in steps:
                q = arrays[0]
                out, lse = torch.empty_like(q), torch.empty((q.shape[0], 8), device="cuda")
                ws = torch.empty(kvattn.attn_workspace_bytes(dp.pool, 8, arrays[5].numel(), int(q.shape[0]), bounds[1]), dtype=torch.uint8,
                                 device="cuda")
                kvattn.attn_extend_append(dp.pool, *[t.cuda() for t in arrays], *bounds, out, lse, ws)
                torch.cuda.synchronize()
                outs.append((synth.bf16_bits(out), lse.cpu().numpy()))
            image = dp.device_image()
        else:
            host = [[_host(t.cpu(), pinned) for t in arrays] for arrays, _ in steps]
            res = [(_host(torch.full(h[0].shape, float("nan"), dtype=torch.bfloat16), pinned), _host(torch.full((h[0].shape[0], 8), float("nan")), pinned))
                   for h in host]
            size = max(kvattn.attn_extend_host_staging_bytes(dp.pool, 8, h[5].numel(), h[0].shape[0], h[4].shape[1], bounds[1])
                       for h, (_, bounds) in zip(host, steps))
            staging = [torch.empty(size, dtype=torch.uint8, device="cuda") for _ in range(areas)]
            torch.cuda.synchronize()
            for s, (h, (_, bounds)) in enumerate(zip(host, steps)):
                kvattn.attn_extend_host(dp.pool, *h, *bounds, *res[s], staging[s % areas])
            torch.cuda.current_stream().synchronize()
            for s, ((o, l), want) in enumerate(zip(res, outs)):
                assert np.array_equal(synth.bf16_bits(o), want[0]) and np.array_equal(l.numpy(), want[1]), s
            assert all(np.array_equal(x, y) for x, y in zip(dp.device_image(), image))
        assert kvattn.kv_last_async_status(dp.pool) == kvattn.KV_OK
        dp.close()
