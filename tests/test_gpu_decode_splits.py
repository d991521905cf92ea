"""attn_decode over every number of CTAs a (sequence, KV head) can be spread over, at the edges of the runs of pages its
warps take, against the oracle element by element."""
import numpy as np
import pytest
import torch

from paper_2607_23815_b200 import kvattn, synth
from harness import Batch, DualPool, assert_close, run_decode

pytestmark = pytest.mark.gpu


def _check(geom, lens, seed):
    dp = DualPool(geom, sum(synth.pages_needed(max(L, 1), 16) for L in lens) + 2, seed=seed)
    b = Batch(dp, [max(L, 1) for L in lens])
    b.write([(i, 0, L) for i, L in enumerate(lens) if L > 0])
    outs = []
    for impl in (2, 1):
        kvattn.kvattn_set_decode_impl(impl)
        try:
            outs.append(run_decode(dp, b, lens, oracle=(impl == 2)))
        finally:
            kvattn.kvattn_set_decode_impl(0)
    assert_close(outs[0], f"decode splits {lens[:4]}")
    assert np.array_equal(outs[0]["o_bits"], outs[1]["o_bits"]) and np.array_equal(outs[0]["lse_raw"], outs[1]["lse_raw"])
    assert kvattn.kv_last_async_status(dp.pool) == kvattn.KV_OK
    dp.close()


@pytest.mark.parametrize("hq,hkv,d", [(4, 1, 128), (8, 1, 64), (1, 1, 64), (8, 8, 128)])
@pytest.mark.parametrize("pages", [4, 8, 12, 16, 24, 32, 64, 97])
def test_one_sequence_over_clusters_of_every_size(pages, hq, hkv, d):
    # a quarter of the pages is what the number of CTAs may reach: 1, 2, 3, 4, 6, 8 and 16 of them are launched here,
    # with runs of one, two and three pages, a last page of one token, and one that is full
    for n in (16 * pages - 15, 16 * pages):
        _check(synth.Geometry(hq, hkv, d), [n], seed=700 + pages)


@pytest.mark.parametrize("max_ctx,batch", [(3100, 90), (10300, 80), (1000, 90)])
def test_more_clusters_than_the_device_holds(max_ctx, batch):
    # one long sequence sets the split for a batch of short ones (most runs are empty), in several waves of clusters
    rng = np.random.default_rng(max_ctx)
    lens = [max_ctx, 0, 1, 16, 17] + [int(x) for x in rng.integers(1, 120, size=batch - 5)]
    _check(synth.Geometry(32, 8, 128), lens, seed=800)


@pytest.mark.parametrize("d,batch,pages", [(128, 1, 192), (128, 1, 193), (64, 1, 264), (64, 1, 265), (128, 320, 6), (128, 320, 7)])
def test_where_the_default_goes_from_registers_to_the_ring(d, batch, pages):
    # two (64 dims: 2.75) pages per warp of 16 CTAs; a batch of more CTAs than are resident: one page per warp of one
    geom = synth.Geometry(8, 1, d)
    lens = [16 * pages] + [16 * (i % pages) + 1 for i in range(batch - 1)]
    dp = DualPool(geom, sum(synth.pages_needed(L, 16) for L in lens) + 2, seed=pages)
    b = Batch(dp, lens)
    b.write([(i, 0, L) for i, L in enumerate(lens)])
    outs = []
    for impl in (0, 1, 2):
        kvattn.kvattn_set_decode_impl(impl)
        try:
            outs.append(run_decode(dp, b, lens, oracle=(impl == 0)))
        finally:
            kvattn.kvattn_set_decode_impl(0)
    assert_close(outs[0], f"decode of {batch} sequences, {pages} pages")
    for o in outs[1:]:
        assert np.array_equal(outs[0]["o_bits"], o["o_bits"]) and np.array_equal(outs[0]["lse_raw"], o["lse_raw"])
    dp.close()


@pytest.mark.parametrize("hq,hkv,d,batch", [(4, 1, 128, 297), (32, 8, 128, 75), (8, 8, 128, 113), (8, 4, 64, 333), (2, 1, 64, 2000)])
def test_ctas_with_several_short_sequences(hq, hkv, d, batch):
    # two, three and six (sequence, KV head) pairs per CTA, the last CTA not full, runs from none to several pages
    rng = np.random.default_rng(batch)
    lens = [0, 1, 16, 17, 80] + [int(x) for x in rng.integers(1, 80, size=batch - 5)]
    _check(synth.Geometry(hq, hkv, d), lens, seed=batch)


def test_back_to_back_calls_that_depend_on_each_other():
    # The kernel is launched early behind whatever runs before it on the stream: an append, another decode, a fill.
    geom = synth.Geometry(8, 2, 128)
    dp = DualPool(geom, 64, seed=12, with_oracle=False)
    b = Batch(dp, [300, 77])
    b.write([(0, 0, 300), (1, 0, 77)])
    i32 = lambda x: torch.tensor(x, dtype=torch.int32, device="cuda")
    bt, cl = torch.from_numpy(b.block_tables()).cuda(), i32([300, 77])
    q = torch.cat([b.q(0, 299, 300), b.q(1, 76, 77)]).contiguous()
    dec = lambda q_, o_, l_: kvattn.attn_decode(dp.pool, q_, bt, cl, 300, geom.scale, o_, l_, None)
    steps = 6
    ref = [q]
    for _ in range(steps):                                      # each step's output is the next one's query
        o, l = torch.empty_like(q), torch.empty((2, 8), device="cuda")
        dec(ref[-1], o, l)
        torch.cuda.synchronize()
        ref.append(o)
    for _ in range(20):
        got = [torch.full_like(q, float("nan")) for _ in range(steps)]
        lse = torch.empty((2, 8), device="cuda")
        x = q
        for o in got:
            dec(x, o, lse)
            x = o
        torch.cuda.synchronize()
        for o, r in zip(got, ref[1:]):
            assert torch.equal(o.view(torch.int16), r.view(torch.int16))
    dp.close()


@pytest.mark.parametrize("d", [128, 64])
@pytest.mark.parametrize("ctx", [16, 700])
@pytest.mark.parametrize("batch", [1, 18, 19, 37, 38])
def test_one_or_two_blocks_per_sm(batch, ctx, d):
    # batches of about as many blocks as there are SMs, and twice as many (148 on a B200, 8 KV heads), of one CTA per pair and of clusters
    rng = np.random.default_rng(batch)
    _check(synth.Geometry(16, 8, d), [ctx] + [int(x) for x in rng.integers(1, ctx + 1, size=batch - 1)], seed=850 + batch)
