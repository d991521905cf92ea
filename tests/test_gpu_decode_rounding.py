"""A row's largest weight is exactly 1 when P is rounded to bf16: a key that takes much of the weight costs no precision."""
import numpy as np
import pytest
import torch

from paper_2607_23815_b200 import kvattn, synth
from harness import Batch, DualPool

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("d", [128, 64])
@pytest.mark.parametrize("way", ["ring", "registers", "small tiles"])
def test_the_largest_weight_is_not_rounded(way, d):
    # Every key has score 0 and value 0 but one, in a page behind the first of its warp's run (18 pages over six warps, or over
    # the one warp of the small-tile kernel), of score s between 3 and 7.9 binades and value 1: O = 2^s / (n - 1 + 2^s).  The
    # exact result is rounded to bf16 once (half a unit in the last place); the fp32 sums and ex2 add some 1e-6.  A weight
    # 2^s taken against an older maximum is rounded as well, by up to half a unit more.
    geom, n, at = synth.Geometry(32, 8, d), 18 * 16, 2 * 16 + 5
    batch = 25                                                   # 200 (sequence, KV head) pairs: one CTA for each
    dp = DualPool(geom, batch * 18, seed=3, with_oracle=False, fill=0)
    b = Batch(dp, [n] * batch)
    for i in range(batch):
        for h in range(8):
            k0 = kvattn.kv_pool_elem_offset(dp.pool, b.rows[i][at // 16], h, at % 16, 0)
            dp.k_buf[k0] = 0x3F80                                # 1.0
            offs = [kvattn.kv_pool_elem_offset(dp.pool, b.rows[i][at // 16], h, at % 16, x) for x in range(d)]
            dp.v_buf[torch.tensor(offs, device="cuda")] = 0x3F80
    scale = 1.0 / 64
    rng = np.random.default_rng(5)
    q = torch.zeros((batch, 32, d), dtype=torch.bfloat16, device="cuda")
    q[:, :, 0] = torch.from_numpy(rng.uniform(3.0, 7.9, (batch, 32)) * 64 * np.log(2)).cuda().bfloat16()
    w = np.exp(q[:, :, 0].double().cpu().numpy() * scale)
    want = w / (n - 1 + w)
    bt, ctx = torch.from_numpy(b.block_tables()).cuda(), torch.full((batch,), n, dtype=torch.int32, device="cuda")
    out, lse = torch.empty_like(q), torch.empty((batch, 32), device="cuda")
    torch.cuda.synchronize()
    if way == "small tiles":
        kvattn.kvattn_set_extend_impl(1)
        try:
            one = torch.ones(batch, dtype=torch.int32, device="cuda")
            cu = torch.arange(batch + 1, dtype=torch.int32, device="cuda")
            kvattn.attn_extend(dp.pool, q, cu, bt, ctx - one, one, 1, n, scale, out, lse, None)
        finally:
            kvattn.kvattn_set_extend_impl(0)
    else:
        kvattn.kvattn_set_decode_impl(2 if way == "ring" else 1)
        try:
            kvattn.attn_decode(dp.pool, q, bt, ctx, n, scale, out, lse, None)
        finally:
            kvattn.kvattn_set_decode_impl(0)
    torch.cuda.synchronize()
    got = out.double().cpu().numpy()
    half_unit = 2.0 ** (np.floor(np.log2(want)) - 8)             # bf16: eight significant bits
    assert np.all(np.abs(got - want[:, :, None]) <= half_unit[:, :, None] + 1e-5 * want[:, :, None])
    assert np.allclose(lse.cpu().numpy(), np.log(n - 1 + w), atol=1e-5)
    assert kvattn.kv_last_async_status(dp.pool) == kvattn.KV_OK
    dp.close()
