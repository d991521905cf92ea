"""Calls on two streams run side by side where the device has room for both: no call keeps the other's blocks off the SMs while it waits
for what is in front of it, nor by asking for more of an SM than it uses.  Graphs of the same calls, on one stream and on two; what two
streams take over what one takes, the best of several turns (a time, but a ratio of two on the same device)."""
import numpy as np
import pytest
import torch

from paper_2607_23815_b200 import kvattn

pytestmark = pytest.mark.gpu


def _i32(x):
    return torch.tensor(np.asarray(x), dtype=torch.int32, device="cuda")


class _Set:
    """P[i] tokens in the pages of sequence i, E[i] of them new."""

    def __init__(self, hq, hkv, d, P, E, seed):
        n, L, T = len(P), [p + e for p, e in zip(P, E)], sum(E)
        need = [-(-x // 16) for x in L]
        gen = torch.Generator(device="cuda").manual_seed(seed)
        randn = lambda *s: torch.randn(s, generator=gen, device="cuda", dtype=torch.bfloat16)
        self.pages = [torch.zeros((sum(need), hkv, 16, d), device="cuda", dtype=torch.bfloat16) for _ in range(2)]
        self.pool = kvattn.kv_pool_create_ex(sum(need), 16, hkv, d, *self.pages)
        ids, bt = np.random.default_rng(seed).permutation(sum(need)).astype(np.int32), np.full((n, max(need)), -1, np.int32)
        for i, k in enumerate(need):
            bt[i, :k], ids = ids[:k], ids[k:]
        self.bt, self.cu, self.pl, self.el, self.ctx = _i32(bt), _i32(np.concatenate([[0], np.cumsum(E)])), _i32(P), _i32(E), _i32(L)
        self.me, self.ml, self.scale = max(E), max(L), d ** -0.5
        self.k, self.v = randn(T, hkv, d), randn(T, hkv, d)
        self.q, self.qd = randn(T, hq, d), randn(n, hq, d)
        self.res = [torch.empty_like(self.q), torch.empty((T, hq), device="cuda")]
        self.resd = [torch.empty_like(self.qd), torch.empty((n, hq), device="cuda")]
        self.ws = torch.empty(max(256, kvattn.attn_workspace_bytes(self.pool, hq, n, T, self.ml, n, self.ml)), dtype=torch.uint8, device="cuda")

    def append(self):
        kvattn.kv_append(self.pool, self.k, self.v, self.cu, self.pl, None, self.bt)

    def decode(self):
        kvattn.attn_decode(self.pool, self.qd, self.bt, self.ctx, self.ml, self.scale, *self.resd, self.ws)

    def extend_append(self):
        kvattn.attn_extend_append(self.pool, self.q, self.k, self.v, self.cu, self.bt, self.pl, self.el, self.me, self.ml, self.scale, *self.res, self.ws)


def _two_over_one(sets, call, calls=20, turns=12):
    side = torch.cuda.Stream()

    def one():
        for i in range(calls):
            for half in range(2):
                call(sets[2 * half + i % 2])

    def two():
        main = torch.cuda.current_stream()
        side.wait_stream(main)
        with torch.cuda.stream(side):
            for i in range(calls):
                call(sets[2 + i % 2])
        for i in range(calls):
            call(sets[i % 2])
        main.wait_stream(side)

    best, graphs = [], []
    for steps in (one, two):
        steps()
        torch.cuda.synchronize()
        graphs.append(torch.cuda.CUDAGraph())
        with torch.cuda.graph(graphs[-1]):
            steps()
    for g in graphs:
        times = []
        for _ in range(turns):
            a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            g.replay()
            a.record()
            for _ in range(5):
                g.replay()
            b.record()
            torch.cuda.synchronize()
            times.append(a.elapsed_time(b))
        best.append(min(times))
    return best[1] / best[0]


def _check(geom, P, E, call, limit):
    sets = [_Set(*geom, P, E, seed) for seed in range(4)]
    ratio = 2.0
    for _ in range(4):  # (some captures put both streams' kernels into one queue of the device)
        ratio = min(ratio, _two_over_one(sets, call))
        if ratio < limit:
            break
    assert all(kvattn.kv_last_async_status(s.pool) == kvattn.KV_OK for s in sets)
    for s in sets:
        kvattn.kv_pool_destroy(s.pool)
    assert ratio < limit, ratio


# (0.90 and 0.91 where the blocks of the next call's append sit on the SMs while they wait, 0.71 and 0.72 where they come at its end)
@pytest.mark.parametrize("geom,P,E", [((16, 4, 128), [850] * 20, [29] * 20), ((32, 8, 128), [950] * 14, [58] * 14)])
def test_extends(geom, P, E):
    _check(geom, P, E, _Set.extend_append, 0.8)


# (0.66, 0.83 and 0.82 where an append's block keeps its SM to itself, 0.52, 0.57 and 0.56 where two share one)
@pytest.mark.parametrize("geom,P,E,limit", [((32, 8, 128), [37] * 3, [60, 60, 28], 0.6), ((16, 2, 128), [37] * 20, [59] * 20, 0.7), ((8, 1, 128), [149] * 148, [1] * 148, 0.7)])
def test_appends(geom, P, E, limit):
    _check(geom, P, E, _Set.append, limit)


# (0.90, 0.97 and 0.91 where blocks ask for an SM to themselves, 0.57, 0.60 and 0.55 where not)
@pytest.mark.parametrize("geom,P", [((32, 8, 128), [39] * 18), ((32, 8, 128), [149] * 9), ((32, 8, 64), [39] * 18)])
def test_decodes(geom, P):
    _check(geom, P, [1] * len(P), _Set.decode, 0.75)
