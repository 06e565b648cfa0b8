"""What is timed: the work a serving engine has this library do in the decode phase, through the
public entry points of ``binding.py``.

Every case is one attention layer's share of one step over a batch of independent requests that
share a paged pool of latent rows (128 heads, or a tensor-parallel shard of them), as
``workloads.py`` describes it:

``decode``       attention over an index list (``select``: whole ``pages``, or ``all`` tokens) of a
                 bf16 or an 8-bit cache; ``entry`` says how the caller issues it: a prepared launch
                 plan, one ordinary call, or a call whose per-step tensors live in host memory
``topk_decode``  the selection producer followed by the attention over what it selected
``sink_recent``  attention sink + recent tokens given as two ranges
``rolling``      the step of a compressed layer: append one row per request, then attend
``quantize``     writing prefill rows into the 8-bit cache

Context lengths are spread evenly over [ctx_min, ctx_max] and dealt out to the requests by the
seed, so a case does the same amount of work whatever the seed; they need not fill a page.
Values are bf16 0.5 * N(0, 1), selection scores N(0, 1).
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2511_22481_b200 import binding as B
from paper_2511_22481_b200 import workloads as W

PAGE, D_QK, D_V = W.PAGE, W.D_QK, W.D_V


def listed():
    return [
        # one user, a shard of 16 heads (tensor parallel over eight GPUs), short context: the
        # smallest call there is, all latency
        dict(name="one_request_16_heads", kind="decode", batch=1, heads=16, ctx_min=4096, ctx_max=4096,
             select="pages", pages=13, cache="bf16", entry="call"),
        # one user with a long document: a single request has to fill the chip
        dict(name="one_request_long", kind="decode", batch=1, heads=128, ctx_min=65536, ctx_max=65536,
             select="pages", pages=128, cache="bf16", entry="plan"),
        # the ordinary data-parallel decode step: page 0, the last 512 tokens, 24 other pages
        dict(name="pages_batch32", kind="decode", batch=32, heads=128, ctx_min=32768, ctx_max=32768,
             select="pages", pages=33, cache="bf16", entry="plan"),
        # a full batch of users at all stages of their contexts, an eighth of each one's pages
        dict(name="pages_ragged_batch128", kind="decode", batch=128, heads=128, ctx_min=4096, ctx_max=65536,
             select="pages", pages=0, cache="bf16", entry="plan"),
        # half of the heads (tensor parallel over two GPUs), a middling batch of odd lengths
        dict(name="pages_64_heads_batch64", kind="decode", batch=64, heads=64, ctx_min=20011, ctx_max=45003,
             select="pages", pages=33, cache="bf16", entry="plan"),
        # token-level sparsity over long contexts: score -> top-k -> attention, every step
        dict(name="topk_batch16", kind="topk_decode", batch=16, heads=128, ctx_min=131072, ctx_max=131072,
             k=2048, entry="plan"),
        # a layer that stays uncompressed: every token attended to
        dict(name="all_tokens_batch32", kind="decode", batch=32, heads=128, ctx_min=65536, ctx_max=65536,
             select="all", pages=0, cache="bf16", entry="plan"),
        # a layer compressed to sink + recent tokens over the ordinary cache; windows start anywhere
        dict(name="sink_recent_batch32", kind="sink_recent", batch=32, heads=128, ctx_min=3001, ctx_max=32805,
             n_sink=64, n_recent=2048),
        # the same layer on a rolling cache that holds nothing else, with the step's append
        dict(name="rolling_batch128", kind="rolling", batch=128, heads=128, ctx_min=2999, ctx_max=1000003,
             n_sink=64, n_recent=1024),
        # the ordinary step over the 8-bit cache
        dict(name="q8_batch32", kind="decode", batch=32, heads=128, ctx_min=32768, ctx_max=32768,
             select="pages", pages=33, cache="q8", entry="call"),
        # a prefill chunk (sixteen prompts of 3.5K tokens) written to the 8-bit cache
        dict(name="quantize_prefill", kind="quantize", rows=57344),
        # the ordinary step for an engine whose activations arrive and leave through host memory
        dict(name="host_batch32", kind="decode", batch=32, heads=128, ctx_min=32768, ctx_max=32768,
             select="pages", pages=33, cache="bf16", entry="host"),
    ]


# No drawn case attends to as many tokens as the largest listed one, or holds more of them.
MOST_TOKENS = 30 * 65536
MOST_POOL_TOKENS = 4_500_000


def _log_int(rng, lo, hi):
    return min(hi, max(lo, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def _contexts(rng, batch, most):
    """(ctx_min, ctx_max): one length for all or a spread, neither a multiple of the page size in general."""
    top = max(1024, min(most, MOST_POOL_TOKENS // batch))
    hi = _log_int(rng, 1024, top)
    return (hi, hi) if rng.random() < 0.3 else (_log_int(rng, max(512, hi // 16), hi), hi)


def draw(rng):
    kind = rng.choice(("decode",) * 6 + ("topk_decode", "topk_decode", "sink_recent", "rolling", "quantize"))
    if kind == "quantize":
        return dict(kind=kind, rows=_log_int(rng, 8192, 262144))
    heads = rng.choice((8, 16, 32, 40, 64, 65, 80, 96, 128, 128, 128, 128))
    if kind == "topk_decode":
        batch = _log_int(rng, 1, 48)
        lo, hi = _contexts(rng, batch, 131072)
        return dict(kind=kind, batch=batch, heads=heads, ctx_min=lo, ctx_max=hi, k=_log_int(rng, 256, min(4096, hi)),
                    entry=rng.choice(("plan", "call")))
    if kind in ("sink_recent", "rolling"):
        batch = _log_int(rng, 1, 160)
        lo, hi = _contexts(rng, batch, 65536)
        if kind == "rolling":
            hi = _log_int(rng, 2048, 1000003)
            lo = _log_int(rng, max(512, hi // 64), hi)
        return dict(kind=kind, batch=batch, heads=heads, ctx_min=lo, ctx_max=hi, n_sink=rng.choice((4, 64, 100, 128)),
                    n_recent=_log_int(rng, 256, 4096))
    batch = _log_int(rng, 1, 256)
    lo, hi = _contexts(rng, batch, 65536)
    cache = rng.choice(("bf16", "bf16", "bf16", "q8"))
    if cache == "q8":
        heads = max(heads, 65)               # the 8-bit path takes more than 64 heads
    select = rng.choice(("pages", "pages", "pages", "all"))
    if select == "all" and batch * hi > MOST_TOKENS:
        select = "pages"
    pages = 0 if rng.random() < 0.25 else _log_int(rng, 9, min(192, MOST_TOKENS // (batch * PAGE)))
    entry = "call" if cache == "q8" else rng.choice(("plan", "plan", "call", "host"))
    return dict(kind="decode", batch=batch, heads=heads, ctx_min=lo, ctx_max=hi, select=select, pages=pages,
                cache=cache, entry=entry)


# ---------------------------------------------------------------------------------------
# sizes that follow from a case alone
# ---------------------------------------------------------------------------------------

def _lengths(case):
    """Context length of every request, in increasing order."""
    n, lo, hi = case["batch"], case["ctx_min"], case["ctx_max"]
    return [hi] * n if lo == hi else [lo + (hi - lo) * i // max(1, n - 1) for i in range(n)]


def _pages(tokens):
    return max(1, -(-tokens // PAGE))


def _selected_pages(case, length):
    """(pages selected, how many of them are the most recent ones) of a page-granular selection."""
    have = _pages(length)
    want = min(have, case["pages"] or max(9, round(have / 8)))
    return want, min(want - 1, max(1, want // 4))


def _selected(case, length):
    """Tokens a request of this length attends to."""
    if case["kind"] == "topk_decode":
        return min(case["k"], length)
    if case["kind"] in ("sink_recent", "rolling"):
        return min(length, case["n_sink"] + case["n_recent"])
    if case["select"] == "all":
        return length
    want, _ = _selected_pages(case, length)
    return want * PAGE - (_pages(length) * PAGE - length)       # the last page is always among them


# ---------------------------------------------------------------------------------------
# what a program has in hand before the call
# ---------------------------------------------------------------------------------------

def _normal(shape, gen):
    return torch.empty(shape, dtype=torch.bfloat16, device="cuda").normal_(0.0, 0.5, generator=gen)


def _page_tables(rng, pages):
    """Every request's pages, scattered over one pool that they fill."""
    table = np.full((len(pages), max(pages)), -1, dtype=np.int32)
    pool, at = rng.permutation(sum(pages)).astype(np.int32), 0
    for b, n in enumerate(pages):
        table[b, :n] = pool[at:at + n]
        at += n
    return table


def _index_lists(case, lengths, rng):
    lists = np.full((len(lengths), max(_selected(case, n) for n in lengths)), -1, dtype=np.int32)
    for b, n in enumerate(lengths):
        if case["select"] == "all":
            at = np.arange(n)
        else:
            have = _pages(n)
            want, recent = _selected_pages(case, n)
            middle = 1 + rng.permutation(max(0, have - recent - 1))[: max(0, want - recent - 1)]
            pages = np.concatenate([[0] if have > recent else [], middle, np.arange(have - recent, have)])
            at = (pages[:, None] * PAGE + np.arange(PAGE)).reshape(-1)
            at = at[at < n]
        lists[b, : len(at)] = at
    return lists, np.array([_selected(case, n) for n in lengths], dtype=np.int32)


class _State:
    pass


def prepare(case, seed):
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed)
    s = _State()
    s.kind, s.entry = case["kind"], case.get("entry")
    if s.kind == "quantize":
        s.rows = _normal((case["rows"], D_QK), gen)
        s.codes = torch.empty((case["rows"], B.OMNI_Q8_ROW_BYTES), dtype=torch.uint8, device="cuda")
        s.scales = torch.empty((case["rows"],), dtype=torch.float32, device="cuda")
        return s
    rng = np.random.default_rng(seed)
    lengths = [int(n) for n in rng.permutation(_lengths(case))]
    batch, heads = case["batch"], case["heads"]
    dev = lambda a: torch.from_numpy(a).to("cuda")  # noqa: E731
    if s.kind == "rolling":
        s.sizes = (case["n_sink"], case["n_recent"])
        pages = [B.omni_rolling_pages_per_request(*s.sizes)] * batch
        max_sel = sum(s.sizes)
    else:
        pages = [_pages(n) for n in lengths]
        max_sel = max(_selected(case, n) for n in lengths)
    table = _page_tables(rng, pages)
    s.q, s.kv = _normal((batch, heads, D_QK), gen), _normal((sum(pages), PAGE, D_QK), gen)
    s.table = dev(table)
    if s.kind in ("sink_recent", "rolling"):
        s.sizes = (case["n_sink"], case["n_recent"])
        max_sel = sum(s.sizes)
        s.ctx = dev(np.array(lengths, dtype=np.int32))
        if s.kind == "rolling":
            s.before, s.row = s.ctx - 1, _normal((batch, D_QK), gen)
    elif s.kind == "topk_decode":
        s.k = max_sel
        s.scores = torch.empty((batch, max(lengths)), device="cuda").normal_(generator=gen)
        s.ctx = dev(np.array(lengths, dtype=np.int32))
        s.idx = torch.zeros((batch, s.k), dtype=torch.int32, device="cuda")
        s.len = torch.zeros((batch,), dtype=torch.int32, device="cuda")
    else:
        lists, counts = _index_lists(case, lengths, rng)
        s.idx, s.len = dev(lists), dev(counts)
    s.desc = B.make_desc(batch, heads, sum(pages), table.shape[1], max_sel, W.SCALE)
    s.out = torch.empty((batch, heads, D_V), dtype=torch.bfloat16, device="cuda")
    s.lse = torch.empty((batch, heads), dtype=torch.float32, device="cuda")
    s.workspace = torch.empty((B.omni_sparse_mla_workspace_bytes(s.desc),), dtype=torch.uint8, device="cuda")
    s.status = torch.zeros((1,), dtype=torch.int32, device="cuda")
    if s.entry == "plan":
        s.plan = B.omni_sparse_mla_plan_init(s.desc, s.q, s.kv)
    elif s.entry == "host":
        pinned = lambda t: t.cpu().pin_memory()  # noqa: E731
        s.q, s.table, s.idx, s.len, s.out, s.lse = (pinned(t) for t in (s.q, s.table, s.idx, s.len, s.out, s.lse))
        s.staging = torch.empty((B.omni_sparse_mla_host_staging_bytes(s.desc),), dtype=torch.uint8, device="cuda")
    if case.get("cache") == "q8":
        s.entry = "q8"
        bf16, rows = s.kv, s.kv.shape[0] * PAGE
        s.kv = torch.empty((s.kv.shape[0], PAGE, B.OMNI_Q8_ROW_BYTES), dtype=torch.uint8, device="cuda")
        s.scales = torch.empty((rows,), dtype=torch.float32, device="cuda")
        B.omni_kv_quantize_q8(bf16, s.kv, s.scales)
    return s


def run(s):
    if s.kind == "quantize":
        B.omni_kv_quantize_q8(s.rows, s.codes, s.scales)
        return s.codes, s.scales
    if s.kind == "rolling":
        B.omni_kv_append_rolling(s.desc, s.kv, s.table, s.before, s.row, *s.sizes, s.status)
        B.omni_sparse_mla_decode_rolling(s.desc, s.q, s.kv, s.table, s.ctx, *s.sizes, s.out, s.lse, s.workspace, s.status)
        return s.out, s.lse, s.kv
    if s.kind == "sink_recent":
        B.omni_sparse_mla_decode_sink_recent(s.desc, s.q, s.kv, s.table, s.ctx, *s.sizes, s.out, s.lse, s.workspace, s.status)
        return s.out, s.lse
    if s.kind == "topk_decode":
        B.omni_topk_select(s.scores, s.ctx, s.k, s.idx, s.len)
    if s.entry == "plan":
        B.omni_sparse_mla_decode_planned(s.plan, s.table, s.idx, s.len, s.out, s.lse, s.workspace, s.status)
    elif s.entry == "call":
        B.omni_sparse_mla_decode(s.desc, s.q, s.kv, s.table, s.idx, s.len, s.out, s.lse, s.workspace, s.status)
    elif s.entry == "q8":
        B.omni_sparse_mla_decode_q8(s.desc, s.q, s.kv, s.scales, s.table, s.idx, s.len, s.out, s.lse, s.workspace, s.status)
    else:
        B.omni_sparse_mla_decode_host(s.desc, s.q, s.kv, s.table, s.idx, s.len, s.out, s.lse, s.staging, s.workspace, s.status)
    if s.kind == "topk_decode":
        return s.out, s.lse, s.idx, s.len
    return s.out, s.lse


def work(case):
    """Each selected cache row, q, the indices or scores read once; the results written once."""
    if case["kind"] == "quantize":
        return {"bytes": case["rows"] * (D_QK * 2 + B.OMNI_Q8_ROW_BYTES + 4), "flops": 0}
    lengths = _lengths(case)
    tokens = sum(_selected(case, n) for n in lengths)
    batch, heads = case["batch"], case["heads"]
    row = B.OMNI_Q8_ROW_BYTES + 4 if case.get("cache") == "q8" else D_QK * 2
    nbytes = tokens * row + batch * heads * ((D_QK + D_V) * 2 + 4)
    nbytes += tokens // PAGE * 4                                    # page ids
    if case["kind"] == "topk_decode":
        nbytes += 4 * sum(lengths) + 2 * 4 * tokens                 # scores; positions written, then read
    elif case["kind"] == "decode":
        nbytes += 4 * tokens
    elif case["kind"] == "rolling":
        nbytes += batch * 2 * D_QK * 2
    return {"bytes": nbytes, "flops": 2 * heads * (D_QK + D_V) * tokens}


def tolerance(case):
    if case["kind"] == "quantize":
        return "exact"
    # out is bf16 and the weights are rounded to bf16 (or as many bits) before the weighted sum: each
    # of the two costs about 2^-9 of the result's norm; positions and cache rows are whole values
    return {"rel": 1e-2, "max": 5e-2, "differ": 0.0}
