"""attn_extend_shared where a parent's and its children's pages share KV steps: page and tile edges, children of one token,
children longer than a tile, items with one step and items split over a cluster of CTAs, against the oracle."""
import numpy as np
import pytest
import torch

from paper_2607_23815_b200 import kvattn, synth
from oracle import paged_attention as orc
from harness import Batch, DualPool, assert_close

pytestmark = pytest.mark.gpu


def _run(geom, parent_lens, child_lens, n_child, seed, small_workspace=False):
    """child_lens: all children's, in the parents' order; n_child: children per parent."""
    pages = sum(synth.pages_needed(L, 16) for L in parent_lens + child_lens) + 4
    dp = DualPool(geom, pages, seed=seed)
    parents, children = Batch(dp, parent_lens, uid0=0), Batch(dp, child_lens, uid0=1000)
    parents.write([(i, 0, L) for i, L in enumerate(parent_lens) if L])
    children.write([(i, 0, L) for i, L in enumerate(child_lens) if L])
    cu_q, cu_c = np.concatenate([[0], np.cumsum(child_lens)]), np.concatenate([[0], np.cumsum(n_child)])
    q = torch.cat([children.q(c, 0, L) for c, L in enumerate(child_lens) if L]).contiguous()
    hq, i32 = geom.n_q_heads, lambda x: torch.tensor(np.asarray(x), dtype=torch.int32, device="cuda")
    rows = [int(cu_q[cu_c[g + 1]] - cu_q[cu_c[g]]) for g in range(len(parent_lens))]
    size = kvattn.attn_extend_shared_workspace_bytes(dp.pool, hq, len(parent_lens), len(child_lens), int(q.shape[0]), max(parent_lens))
    if small_workspace:  # what the call needs without partial results: the merged copies and the item list
        size = 4 * (2 * len(parent_lens) + 1 + len(child_lens)) + q.numel() * 2 + q.shape[0] * hq * 4 + 32 * (q.shape[0] // 32 + len(child_lens) + 2) + 4096
    out, lse = torch.full_like(q, float("nan")), torch.full((q.shape[0], hq), float("nan"), device="cuda")
    kvattn.attn_extend_shared(dp.pool, q, i32(cu_q), i32(cu_c), i32(parents.block_tables()), i32(parent_lens),
                              i32(children.block_tables()), i32(child_lens), max(child_lens), max(rows), max(parent_lens), geom.scale,
                              out, lse, torch.empty(size, dtype=torch.uint8, device="cuda"))
    torch.cuda.synchronize()
    assert kvattn.kv_last_async_status(dp.pool) == kvattn.KV_OK
    o_ref, l_ref = orc.attn_extend_shared(dp.host, synth.bf16_bits(q), hq, cu_q.astype(np.int32), cu_c.astype(np.int32),
                                          parents.block_tables(), parent_lens, children.block_tables(), child_lens, geom.scale)
    assert_close({"o": out.float().cpu().numpy().astype(np.float64), "lse": lse.cpu().numpy().astype(np.float64), "o_ref": o_ref,
                  "lse_ref": l_ref}, f"fan-out {parent_lens[:3]} {child_lens[:5]}")
    dp.close()


@pytest.mark.parametrize("hq,hkv,d", [(8, 2, 128), (16, 2, 64), (2, 2, 128)])
@pytest.mark.parametrize("parent", [0, 16, 112, 128, 144, 504, 1040])
def test_one_parent_at_page_and_step_edges(parent, hq, hkv, d):
    # children that end inside a page, on it, take one token, several pages, more than a tile; the parent ends a step,
    # leaves room in it for one page, or for seven.  One parent's items are few: they are split over clusters of CTAs.
    _run(synth.Geometry(hq, hkv, d), [parent], [1, 16, 17, 40, 0, 3, 130, 15], [8], 1100 + parent)
    _run(synth.Geometry(hq, hkv, d), [parent], [1] * 50, [50], 1200 + parent)


@pytest.mark.parametrize("small_workspace", [False, True])
def test_many_parents_with_children_of_every_length(small_workspace):
    rng = np.random.default_rng(12)
    parent_lens = [int(x) * 16 for x in rng.integers(0, 40, size=60)]
    n_child = [int(x) for x in rng.integers(0, 9, size=60)]
    n_child[3], n_child[59] = 1, 2
    child_lens = [int(x) for x in rng.integers(0, 50, size=sum(n_child))]
    child_lens[-1] = 300
    _run(synth.Geometry(8, 2, 128), parent_lens, child_lens, n_child, 1300, small_workspace)
