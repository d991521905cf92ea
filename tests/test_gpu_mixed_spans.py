"""attn_mixed with an extend set that is cut into spans: several spans per CTA, and a decode set that is refused."""
import numpy as np
import pytest
import torch

from paper_2607_23815_b200 import kvattn, synth
from harness import Batch, DualPool, assert_close, extend_schedule, run_extend

pytestmark = pytest.mark.gpu


def _i32(x):
    return torch.tensor(np.asarray(x), dtype=torch.int32, device="cuda")


class _Step:
    """40 sequences of one tile pair, two of them of 24 KV steps, 2 KV heads: spans, and the long items are cut several times."""

    def __init__(self, d, seed, oracle=False):
        self.geom = synth.Geometry(8, 2, d)
        self.P, self.E = [2950] + [40] * 18 + [2939] + [130] * 20, [50] + [20] * 18 + [61] + [33] * 20
        L = [p + e for p, e in zip(self.P, self.E)]
        self.dp = DualPool(self.geom, sum(synth.pages_needed(x, 16) for x in L) + 2, seed=seed, with_oracle=oracle)
        self.b = Batch(self.dp, L)
        self.b.write([(i, 0, x) for i, x in enumerate(L)])
        self.ml, self.me, self.hq = max(L), max(self.E), 8
        self.q = torch.cat([self.b.q(i, self.P[i], L[i]) for i in range(len(L))]).contiguous()
        self.bt, self.cu = torch.from_numpy(self.b.block_tables()).cuda(), _i32(np.concatenate([[0], np.cumsum(self.E)]))
        self.pl, self.el = _i32(self.P), _i32(self.E)
        self.rows = [0, 19, 25]                                     # the decode set: three of the same sequences
        self.qd, self.ctx, self.btd = self.q[:3].contiguous(), _i32([L[i] for i in self.rows]), self.bt[self.rows].contiguous()
        n = kvattn.attn_workspace_bytes(self.dp.pool, 8, len(L), int(self.q.shape[0]), self.ml, 3, self.ml)
        self.ws = torch.empty(n, dtype=torch.uint8, device="cuda")
        assert extend_schedule(self.dp.pool, 8, self.q, self.cu, self.bt, self.pl, self.el, self.me, self.ml, self.geom.scale, self.ws) == "spans"

    def results(self):
        return torch.full_like(self.q, float("nan")), torch.full((self.q.shape[0], 8), float("nan"), device="cuda")

    def plain(self):
        out, lse = self.results()
        kvattn.attn_extend(self.dp.pool, self.q, self.cu, self.bt, self.pl, self.el, self.me, self.ml, self.geom.scale, out, lse, self.ws)
        torch.cuda.synchronize()
        return out, lse

    def mixed(self, max_ctx=None):
        out, lse = self.results()
        od, ld = torch.empty_like(self.qd), torch.empty((3, 8), device="cuda")
        ea = kvattn.extend_args(self.q, self.cu, self.bt, self.pl, self.el, self.me, self.ml, out, lse)
        da = kvattn.decode_args(self.qd, self.btd, self.ctx, max_ctx or self.ml, od, ld)
        try:
            kvattn.attn_mixed(self.dp.pool, 8, self.geom.scale, ea, da, self.ws)
            status = kvattn.KV_OK
        except kvattn.KvError as e:
            status = e.status
        torch.cuda.synchronize()
        return status, out, lse, od, ld


@pytest.mark.parametrize("d", [128, 64])
def test_an_extend_set_is_whole_even_if_the_decode_set_is_refused(d):
    s = _Step(d, seed=81)
    want = s.plain()
    status, out, lse, _, _ = s.mixed(max_ctx=s.bt.shape[1] * 16 + 1)      # longer than the tables
    assert status == kvattn.KV_ERR_INVALID
    assert torch.equal(out.view(torch.int16), want[0].view(torch.int16)) and torch.equal(lse, want[1])
    assert kvattn.kv_last_async_status(s.dp.pool) == kvattn.KV_OK
    s.dp.close()


@pytest.mark.parametrize("d", [128, 64])
def test_several_spans_per_cta(d):
    # 148 spans on a B200; shares of 74, 40 and 16 SMs: two, four and nine spans for a CTA (148 is no multiple of nine, so the
    # last CTA has fewer), three and more of them inside one long item
    s = _Step(d, seed=82, oracle=True)
    assert_close(run_extend(s.dp, s.b, s.P, s.E), "spans")
    want, alone = s.plain(), None
    for cap in (148, 74, 40, 16):
        kvattn.kvattn_set_mixed_extend_ctas(cap)
        try:
            status, out, lse, od, ld = s.mixed()
        finally:
            kvattn.kvattn_set_mixed_extend_ctas(0)
        assert status == kvattn.KV_OK
        assert torch.equal(out.view(torch.int16), want[0].view(torch.int16)) and torch.equal(lse, want[1]), cap
        alone = alone or (od, ld)
        assert torch.equal(od.view(torch.int16), alone[0].view(torch.int16)) and torch.equal(ld, alone[1]), cap
    assert kvattn.kv_last_async_status(s.dp.pool) == kvattn.KV_OK
    s.dp.close()
