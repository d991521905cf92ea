"""What a user of the library has it do: pipeline steps over a paged KV pool, from one short answer to a long-document batch.

A case is one call (or the few calls that belong together) of the public binding `paper_2607_23815_b200.kvattn`, with
everything an engine holds beforehand - the pool with the upstream operators' pages in it, block tables, lengths on the
device, queries, new K/V rows, output tensors, the workspace - made by prepare().  Sizes are those of the library's
own workloads (8B and 70B head geometry, tuple contexts of a few hundred to sixteen thousand tokens, operator
instructions of tens to hundreds of tokens), down to the single tuple that is left at the end of a pipeline.

Sequence lengths belong to the case (they are drawn from its `lengths` number); values and the physical page placement
come from the seed.  Values are N(0, 1) in bf16, the distribution of the library's tests and benchmark.
"""
import math
import random

import numpy as np
import torch

from paper_2607_23815_b200 import kvattn

PAGE = 16
SLAB = 1 << 16  # tokens written into the pool by one call while a state is prepared


def _case(name, op, geom, n, prefix=(0, 0), suffix=(0, 0), ctx=(0, 0), n_dec=0, fan=0, layers=1, lengths=1):
    hq, hkv, d = geom
    return {"name": name, "op": op, "hq": hq, "hkv": hkv, "d": d, "n": n, "prefix_lo": prefix[0], "prefix_hi": prefix[1],
            "suffix_lo": suffix[0], "suffix_hi": suffix[1], "n_dec": n_dec, "ctx_lo": ctx[0], "ctx_hi": ctx[1], "fan": fan,
            "layers": layers, "lengths": lengths}


G8B, G70B, G64 = (32, 8, 128), (64, 8, 128), (32, 8, 64)


def listed():
    return [
        # one token of the last tuple's answer: the smallest call there is
        _case("decode_one", "decode", G8B, 0, n_dec=1, ctx=(517, 517), lengths=11),
        # a few answers at the head or the tail of a pipeline, ragged contexts, heads of 64 dims
        _case("decode_few_d64", "decode", G64, 0, n_dec=13, ctx=(200, 3000), lengths=12),
        # the answers of a full batch
        _case("decode_8b", "decode", G8B, 0, n_dec=256, ctx=(1024, 4096), lengths=13),
        # a handful of long documents being answered about
        _case("decode_long_70b", "decode", G70B, 0, n_dec=5, ctx=(8192, 16384), lengths=14),
        # one tuple moves to the next operator: its suffix is stored and attends over the reused pages
        _case("extend_one", "extend_append", G8B, 1, prefix=(1483, 1483), suffix=(37, 37), lengths=15),
        # the headline batch: 64 tuples move to the next operator
        _case("extend_8b", "extend_append", G8B, 64, prefix=(512, 2048), suffix=(64, 256), lengths=16),
        # long-document reuse
        _case("long_doc_70b", "extend", G70B, 32, prefix=(8192, 16384), suffix=(128, 512), lengths=17),
        # the cache-miss path: tuples of the paper's datasets prefilled from scratch
        _case("prefill_8b", "extend_append", G8B, 7, suffix=(419, 2733), lengths=18),
        # one step of two chained operators: new tokens stored, then the extend set and the decode set together
        _case("pipeline_step", "mixed", G8B, 48, prefix=(256, 3072), suffix=(32, 192), n_dec=192, ctx=(512, 4088), lengths=19),
        # a join: every child of a parent attends over the parent's pages and its own suffix
        _case("fanout_8b", "fanout", G8B, 32, prefix=(1920, 2368), suffix=(30, 44), fan=17, lengths=20),
        # a small step through several layers of a model: one plan, then store + attend per layer
        _case("layers_8b", "layers", G8B, 9, prefix=(300, 2000), suffix=(20, 90), layers=4, lengths=21),
        # a step whose inputs and results live in host memory
        _case("host_step_8b", "host", G8B, 16, prefix=(512, 2048), suffix=(64, 256), lengths=22),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    op = rng.choice(["decode", "decode", "extend_append", "extend_append", "extend", "mixed", "fanout", "layers", "host"])
    geom = rng.choice([G8B, G8B, G70B, G64, (8, 8, 128), (16, 8, 64)])
    lengths = rng.randrange(1000, 1 << 30)

    def span(lo, hi):  # a range of lengths
        b = _log_int(rng, lo, hi)
        return (max(lo, int(b * rng.uniform(0.25, 1.0))), b)

    if op == "decode":
        ctx = span(64, 16384)
        return _unnamed(_case("", op, geom, 0, n_dec=_log_int(rng, 1, max(1, min(256, 650000 // ctx[1]))), ctx=ctx, lengths=lengths))
    if op == "mixed":
        n = _log_int(rng, 1, 48)
        return _unnamed(_case("", op, geom, n, prefix=span(64, 3072), suffix=span(16, 192), n_dec=_log_int(rng, 2, 192),
                              ctx=span(128, 4088), lengths=lengths))
    if op == "fanout":
        return _unnamed(_case("", op, geom, _log_int(rng, 1, 32), prefix=span(256, 2368), suffix=span(8, 44),
                              fan=rng.randint(3, 17), lengths=lengths))
    if op == "layers":
        return _unnamed(_case("", op, geom, _log_int(rng, 1, 24), prefix=span(64, 2048), suffix=span(8, 128),
                              layers=rng.randint(2, 4), lengths=lengths))
    if op == "host":
        return _unnamed(_case("", op, geom, _log_int(rng, 1, 24), prefix=span(64, 2048), suffix=span(16, 256), lengths=lengths))
    if op == "extend":
        p = span(2048, 16384)
        return _unnamed(_case("", op, geom, _log_int(rng, 1, 24), prefix=p, suffix=span(16, 400), lengths=lengths))
    if rng.random() < 0.35:  # from scratch
        s = span(64, 4096)
        return _unnamed(_case("", op, geom, _log_int(rng, 1, max(1, min(48, 24000 // s[1]))), suffix=s, lengths=lengths))
    return _unnamed(_case("", op, geom, _log_int(rng, 1, 64), prefix=span(64, 4096), suffix=span(4, 256), lengths=lengths))


def _unnamed(c):
    del c["name"]
    return c


# ---- lengths, work --------------------------------------------------------------------------------------------------
def _lengths(c):
    """(prefix, suffix) of the extend sequences (fan-out: prefix per parent, suffix per child) and the decode contexts."""
    r = random.Random(c["lengths"])
    P = [r.randint(c["prefix_lo"], c["prefix_hi"]) for _ in range(c["n"])]
    if c["op"] == "fanout":  # the part of a parent's prompt that its children share is made of whole pages
        P = [max(PAGE, p // PAGE * PAGE) for p in P]
        E = [r.randint(c["suffix_lo"], c["suffix_hi"]) for _ in range(c["n"] * c["fan"])]
    else:
        E = [r.randint(c["suffix_lo"], c["suffix_hi"]) for _ in range(c["n"])]
    C = [r.randint(c["ctx_lo"], c["ctx_hi"]) for _ in range(c["n_dec"])]
    return P, E, C


def work(c):
    P, E, C = _lengths(c)
    hq, d, kv_tok = c["hq"], c["d"], 2 * c["hkv"] * c["d"] * 2
    row = hq * d * 2 * 2 + hq * 4                                     # Q in, O out, LSE out, per query token
    rows, pairs, tok_bytes = sum(E), 0, 0
    if c["op"] == "fanout":
        for i, e in enumerate(E):
            pairs += e * P[i // c["fan"]] + e * (e + 1) // 2
        tok_bytes = (sum(P) + sum(E)) * kv_tok
    else:
        for p, e in zip(P, E):
            pairs += e * p + e * (e + 1) // 2
        # keys are read once; a suffix that is stored in the same pass comes from the caller's rows and is written once
        stored = 0 if c["op"] == "extend" else sum(E) * kv_tok
        tok_bytes = (sum(P) + sum(E)) * kv_tok + stored
    pairs += sum(C)
    tok_bytes += sum(C) * kv_tok + (2 * len(C) * kv_tok if c["op"] == "mixed" else 0)
    rows += len(C)
    n = c["layers"]
    return {"bytes": n * (tok_bytes + rows * row), "flops": n * 4.0 * d * hq * pairs}


def tolerance(c):
    # O is rounded to bf16 once and P once before P V: against the same sums in 64 bits the relative error (2-norm) of O
    # is 2.2e-3 to 2.4e-3 and its largest single error 0.006 to 0.010 of the result's root mean square, on every op
    return {"rel": 0.01, "max": 0.04}


# ---- states ---------------------------------------------------------------------------------------------------------
def _i32(x):
    return torch.tensor(np.asarray(x), dtype=torch.int32, device="cuda")


class _Maker:
    """Draws values and hands out pages of one pool (or of one pool per layer, all with the same page ids)."""

    def __init__(self, c, seed, n_pages):
        self.c = c
        self.gen = torch.Generator(device="cuda").manual_seed(seed * 1000003 + c["lengths"] % 1000003)
        shape = (n_pages, c["hkv"], PAGE, c["d"])
        self.pages = [tuple(torch.zeros(shape, dtype=torch.bfloat16, device="cuda") for _ in range(2)) for _ in range(c["layers"])]
        self.pools = [kvattn.kv_pool_create_ex(n_pages, PAGE, c["hkv"], c["d"], k, v) for k, v in self.pages]
        ids = [kvattn.kv_alloc(p, n_pages) for p in self.pools][0]
        order = np.random.default_rng(seed).permutation(n_pages)
        self.ids, self.next = np.asarray(ids, dtype=np.int32)[order], 0

    def randn(self, *shape):
        return torch.randn(shape, generator=self.gen, device="cuda", dtype=torch.bfloat16)

    def kv(self, n):
        return self.randn(n, self.c["hkv"], self.c["d"]), self.randn(n, self.c["hkv"], self.c["d"])

    def table(self, lens, width=None):
        need = [-(-n // PAGE) for n in lens]
        bt = np.full((len(lens), width or max(need + [1])), -1, dtype=np.int32)
        for i, k in enumerate(need):
            bt[i, :k] = self.ids[self.next:self.next + k]
            self.next += k
        return torch.from_numpy(bt).cuda()

    def fill(self, bt, lens, rows=None):
        """Writes tokens 0 .. lens[i]-1 of the table's rows (an earlier operator's work)."""
        rows = list(range(len(lens))) if rows is None else rows
        at = 0
        while at < len(lens):
            end, tok = at, 0
            while end < len(lens) and (tok == 0 or tok + lens[end] <= SLAB):
                tok += lens[end]
                end += 1
            if tok:
                cu = _i32(np.concatenate([[0], np.cumsum(lens[at:end])]))
                start, seg = _i32([0] * (end - at)), _i32(rows[at:end])
                for pool in self.pools:
                    k, v = self.kv(tok)
                    kvattn.kv_append(pool, k, v, cu, start, seg, bt)
            at = end


def prepare(c, seed):
    P, E, C = _lengths(c)
    hq, d, op = c["hq"], c["d"], c["op"]
    pg = lambda lens: sum(-(-n // PAGE) for n in lens)  # noqa: E731
    if op == "fanout":
        m = _Maker(c, seed, pg(P) + pg(E))
        return _prepare_fanout(c, m, P, E)
    L = [p + e for p, e in zip(P, E)]
    ctx = [x + 1 for x in C] if op == "mixed" else C                  # a pipeline step adds one token per answer
    m = _Maker(c, seed, pg(L) + pg(ctx))
    s = {"c": c, "pool": m.pools[0], "pools": m.pools, "pages": m.pages, "scale": float(np.float32(1.0 / math.sqrt(d)))}
    if op == "mixed":                                                 # one table: the extend rows, then the decode rows
        bt = m.table(L + ctx)
        bt_e, bt_d = bt[:len(L)], bt[len(L):]
        s["bt"] = bt
    else:
        bt_e = m.table(L) if L else None
        bt_d = m.table(ctx) if ctx else None
    if L:
        m.fill(bt_e, L if op == "extend" else P)                      # "extend": the suffix has been stored already
        s.update(q=m.randn(sum(E), hq, d), cu=_i32(np.concatenate([[0], np.cumsum(E)])), bt_e=bt_e, p=_i32(P), e=_i32(E),
                 max_e=max(E), max_l=max(L))
        s.update(out=torch.zeros_like(s["q"]), lse=torch.zeros(sum(E), hq, device="cuda"))
    if ctx:
        m.fill(bt_d, C)
        s.update(qd=m.randn(len(ctx), hq, d), bt_d=bt_d, ctx=_i32(ctx), max_c=max(ctx))
        s.update(out_d=torch.zeros_like(s["qd"]), lse_d=torch.zeros(len(ctx), hq, device="cuda"))
    new = sum(E) + (len(C) if op == "mixed" else 0)
    if op in ("extend_append", "host", "mixed"):
        s["k_new"], s["v_new"] = m.kv(new)
    if op == "layers":
        s["kv_new"] = [m.kv(new) for _ in range(c["layers"])]
        s["qs"] = [m.randn(sum(E), hq, d) for _ in range(c["layers"])]
        s["outs"] = [(torch.zeros_like(s["q"]), torch.zeros_like(s["lse"])) for _ in range(c["layers"])]
    if op == "mixed":
        s["cu_new"] = _i32(np.concatenate([[0], np.cumsum(E + [1] * len(C))]))
        s["start_new"] = _i32(P + C)
    if op == "host":
        for k in ("q", "k_new", "v_new", "cu", "bt_e", "p", "e"):
            s[k] = s[k].cpu().pin_memory()
        s["out"], s["lse"] = torch.zeros(s["q"].shape, dtype=torch.bfloat16).pin_memory(), torch.zeros(sum(E), hq).pin_memory()
        n = kvattn.attn_extend_host_staging_bytes(m.pools[0], hq, len(E), sum(E), s["bt_e"].shape[1], s["max_l"])
        s["ws"] = torch.empty(n, dtype=torch.uint8, device="cuda")
    else:
        n = kvattn.attn_workspace_bytes(m.pools[0], hq, len(L), sum(E), max(L + [0]), len(ctx), max(ctx + [0]))
        s["ws"] = torch.empty(max(n, 256), dtype=torch.uint8, device="cuda")
    if op == "mixed":
        s["ea"] = kvattn.extend_args(s["q"], s["cu"], bt_e, s["p"], s["e"], s["max_e"], s["max_l"], s["out"], s["lse"])
        s["da"] = kvattn.decode_args(s["qd"], bt_d, s["ctx"], s["max_c"], s["out_d"], s["lse_d"])
    return s


def _prepare_fanout(c, m, P, E):
    hq, d, fan = c["hq"], c["d"], c["fan"]
    pt, ct = m.table(P), m.table(E)
    m.fill(pt, P)
    m.fill(ct, E)
    s = {"c": c, "pool": m.pools[0], "pools": m.pools, "pages": m.pages, "scale": float(np.float32(1.0 / math.sqrt(d))),
         "q": m.randn(sum(E), hq, d), "cu": _i32(np.concatenate([[0], np.cumsum(E)])), "cu_children": _i32(np.arange(len(P) + 1) * fan),
         "pt": pt, "ct": ct, "p": _i32(P), "e": _i32(E), "max_e": max(E), "max_p": max(P),
         "max_rows": max(sum(E[g * fan:(g + 1) * fan]) for g in range(len(P)))}
    s.update(out=torch.zeros_like(s["q"]), lse=torch.zeros(sum(E), hq, device="cuda"))
    n = kvattn.attn_extend_shared_workspace_bytes(m.pools[0], hq, len(P), len(E), sum(E), max(P))
    s["ws"] = torch.empty(max(n, 256), dtype=torch.uint8, device="cuda")
    return s


# ---- one pass -------------------------------------------------------------------------------------------------------
def run(s):
    c, pool, op = s["c"], s["pool"], s["c"]["op"]
    if op == "decode":
        kvattn.attn_decode(pool, s["qd"], s["bt_d"], s["ctx"], s["max_c"], s["scale"], s["out_d"], s["lse_d"], s["ws"])
        return s["out_d"], s["lse_d"]
    if op == "extend_append":
        kvattn.attn_extend_append(pool, s["q"], s["k_new"], s["v_new"], s["cu"], s["bt_e"], s["p"], s["e"], s["max_e"], s["max_l"],
                                  s["scale"], s["out"], s["lse"], s["ws"])
        return s["out"], s["lse"], s["pages"]
    if op == "extend":
        kvattn.attn_extend(pool, s["q"], s["cu"], s["bt_e"], s["p"], s["e"], s["max_e"], s["max_l"], s["scale"], s["out"], s["lse"],
                           s["ws"])
        return s["out"], s["lse"]
    if op == "mixed":
        kvattn.kv_append(pool, s["k_new"], s["v_new"], s["cu_new"], s["start_new"], None, s["bt"])
        kvattn.attn_mixed(pool, c["hq"], s["scale"], s["ea"], s["da"], s["ws"])
        return s["out"], s["lse"], s["out_d"], s["lse_d"], s["pages"]
    if op == "fanout":
        kvattn.attn_extend_shared(pool, s["q"], s["cu"], s["cu_children"], s["pt"], s["p"], s["ct"], s["e"], s["max_e"], s["max_rows"],
                                  s["max_p"], s["scale"], s["out"], s["lse"], s["ws"])
        return s["out"], s["lse"]
    if op == "layers":
        kvattn.attn_extend_plan(pool, c["hq"], s["cu"], s["bt_e"], s["p"], s["e"], s["q"].shape[0], s["max_e"], s["max_l"], s["ws"])
        for layer, q, (k, v), (out, lse) in zip(s["pools"], s["qs"], s["kv_new"], s["outs"]):
            kvattn.kv_append(layer, k, v, s["cu"], s["p"], None, s["bt_e"])
            kvattn.attn_extend_planned(layer, q, s["cu"], s["bt_e"], s["p"], s["e"], s["max_e"], s["max_l"], s["scale"], out, lse,
                                       s["ws"])
        return s["outs"], s["pages"]
    if op == "host":
        kvattn.attn_extend_host(pool, s["q"], s["k_new"], s["v_new"], s["cu"], s["bt_e"], s["p"], s["e"], s["max_e"], s["max_l"],
                                s["scale"], s["out"], s["lse"], s["ws"])
        return s["out"], s["lse"], s["pages"]
    raise ValueError(op)
