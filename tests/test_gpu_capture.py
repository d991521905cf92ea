"""Steps captured into CUDA graphs: library kernels behind copies, fills and joins of other streams, and behind each other; every
replay with other inputs gives the bits of the calls themselves."""
import numpy as np
import pytest
import torch

from paper_2607_23815_b200 import kvattn, synth
from harness import Batch, DualPool

pytestmark = pytest.mark.gpu


def _i32(x):
    return torch.tensor(np.asarray(x), dtype=torch.int32, device="cuda")


@pytest.mark.parametrize("front", ["copy", "fill", "join", "nothing"])
@pytest.mark.parametrize("P,E", [([1400], [30]), ([2950] + [40] * 18 + [2939] + [130] * 20, [50] + [20] * 18 + [61] + [33] * 20), ([300] * 60, [70] * 60)])
def test_a_captured_step(P, E, front):
    # one sequence (clusters), long among short ones (spans), a full batch (the list); then a mixed step and a decode call
    geom, hq, B, T = synth.Geometry(8, 2, 128), 8, len(P), sum(E)
    L = [p + e for p, e in zip(P, E)]
    dp = DualPool(geom, sum(synth.pages_needed(x, 16) for x in L) + 2, seed=55, with_oracle=False)
    b = Batch(dp, L)
    b.write([(i, 0, P[i]) for i in range(B)])
    gen = torch.Generator(device="cuda").manual_seed(5)
    randn = lambda *s: torch.randn(s, generator=gen, device="cuda", dtype=torch.bfloat16)
    sets = [(randn(T, hq, 128), randn(T, 2, 128), randn(T, 2, 128)) for _ in range(3)]
    q, k, v = (t.clone() for t in sets[0])
    bt, cu, pl, el, ctx, ml = torch.from_numpy(b.block_tables()).cuda(), _i32(np.concatenate([[0], np.cumsum(E)])), _i32(P), _i32(E), _i32(L), max(L)
    ws = torch.empty(kvattn.attn_workspace_bytes(dp.pool, hq, B, T, ml, B, ml), dtype=torch.uint8, device="cuda")
    qd, scratch = randn(B, hq, 128), torch.empty(1 << 20, dtype=torch.uint8, device="cuda")
    new = lambda *s: torch.full(s, 7.0, device="cuda")
    res = [(new(T, hq, 128).bfloat16(), new(T, hq)) for _ in range(3)] + [(new(B, hq, 128).bfloat16(), new(B, hq)) for _ in range(2)]
    side = torch.cuda.Stream()

    def between():
        if front == "copy":
            scratch[:4096].copy_(scratch[4096:8192])
        elif front == "fill":
            scratch.zero_()
        elif front == "join":
            main = torch.cuda.current_stream()
            side.wait_stream(main)
            with torch.cuda.stream(side):
                scratch.zero_()
            main.wait_stream(side)

    def step():
        between()
        kvattn.kv_append(dp.pool, k, v, cu, pl, None, bt)
        between()
        kvattn.attn_extend(dp.pool, q, cu, bt, pl, el, max(E), ml, geom.scale, *res[0], ws)
        between()
        kvattn.attn_extend_append(dp.pool, q, k, v, cu, bt, pl, el, max(E), ml, geom.scale, *res[1], ws)
        between()
        kvattn.attn_mixed(dp.pool, hq, geom.scale, kvattn.extend_args(q, cu, bt, pl, el, max(E), ml, *res[2]),
                          kvattn.decode_args(qd, bt, ctx, ml, *res[3]), ws)
        between()
        kvattn.attn_decode(dp.pool, qd, bt, ctx, ml, geom.scale, *res[4], ws)

    def results():
        torch.cuda.synchronize()
        return [(o.clone().view(torch.int16), l.clone()) for o, l in res]

    def load(s):
        for t, x in zip((q, k, v), sets[s]):
            t.copy_(x)

    want = []
    for s in range(3):
        load(s)
        step()
        want.append(results())
    stream, graph = torch.cuda.Stream(), torch.cuda.CUDAGraph()
    torch.cuda.synchronize()
    with torch.cuda.graph(graph, stream=stream):
        step()
    for s in (1, 2, 0, 0):
        for o, l in res:
            o.fill_(7.0)
            l.fill_(7.0)
        load(s)
        graph.replay()
        for (o, l), (wo, wl) in zip(results(), want[s]):
            assert torch.equal(o, wo) and torch.equal(l, wl), s
    assert kvattn.kv_last_async_status(dp.pool) == kvattn.KV_OK
    del graph
    dp.close()
