"""A last wave of a few requests runs in pieces: whole requests, cut ones, short and empty ones all come out as in
a run without any split.

Bound: either result differs from exact attention by at most 2e-3 + 2^-8 |o| per element (bf16 weights and
results), so the two differ by at most twice that; the log-sum-exps of either are within 2e-3."""
import math

import pytest
import torch

from paper_2511_22481_b200 import binding as B

pytestmark = pytest.mark.gpu
PAGES = 66


def _problem(batch, heads, ragged, seed):
    gen = torch.Generator(device="cuda").manual_seed(seed)
    kv = torch.empty((batch * PAGES, 64, 576), device="cuda", dtype=torch.bfloat16).normal_(0, 0.5, generator=gen)
    q = torch.empty((batch, heads, 576), device="cuda", dtype=torch.bfloat16).normal_(0, 0.5, generator=gen)
    table = torch.randperm(batch * PAGES, device="cuda", generator=gen).to(torch.int32).view(batch, PAGES)
    ctx = torch.full((batch,), PAGES * 64, dtype=torch.int32, device="cuda")
    if ragged:
        # "long": the requests left over are cut, one of them empty; "any": they run beside the longest ones
        least = 1 if ragged == "any" else PAGES * 48
        ctx = torch.randint(least, PAGES * 64 + 1, (batch,), device="cuda", generator=gen).to(torch.int32)
        ctx[batch // 2], ctx[-1] = 0, PAGES * 64
    return q, kv, table, ctx


@pytest.mark.parametrize("batch,heads,ragged,form", [
    (75, 128, None, "list"),       # one request left over
    (80, 128, "long", "list"), (98, 128, "long", "list"), (80, 128, "any", "list"), (98, 128, "any", "q8"), (98, 65, None, "list"), (80, 40, "long", "list"),
    (80, 128, "long", "ranges"), (98, 128, None, "ranges"),
    (80, 128, "long", "q8"), (98, 128, "long", "q8"),
])
def test_tail_in_pieces_equals_whole(batch, heads, ragged, form):
    q, kv, table, ctx = _problem(batch, heads, ragged, 7 * batch + heads)
    limit = PAGES * 64
    idx = torch.arange(limit, dtype=torch.int32, device="cuda").expand(batch, -1).contiguous()
    if form == "q8":
        codes = torch.empty((batch * PAGES, 64, 640), dtype=torch.uint8, device="cuda")
        scale = torch.empty((batch * PAGES * 64,), device="cuda")
        B.omni_kv_quantize_q8(kv.view(-1, 576), codes.view(-1, 640), scale)
    results = []
    for splits in (0, 1):
        d = B.make_desc(batch, heads, batch * PAGES, PAGES, limit, 1.0 / math.sqrt(192.0), num_splits=splits)
        assert B.omni_sparse_mla_num_launches(d) == (2 if splits == 0 else 1)
        ws = torch.full((B.omni_sparse_mla_workspace_bytes(d),), 255, dtype=torch.uint8, device="cuda")
        out = torch.full((batch, heads, 512), float("nan"), dtype=torch.bfloat16, device="cuda")
        lse = torch.full((batch, heads), float("nan"), device="cuda")
        status = torch.zeros(1, dtype=torch.int32, device="cuda")
        for _ in range(2):             # a second step finds the first one's workspace
            if form == "q8":
                B.omni_sparse_mla_decode_q8(d, q, codes, scale, table, idx, ctx, out, lse, ws, status)
            elif form == "ranges":
                B.omni_sparse_mla_decode_sink_recent(d, q, kv, table, ctx, 64, limit - 64, out, lse, ws, status)
            else:
                B.omni_sparse_mla_decode(d, q, kv, table, idx, ctx, out, lse, ws, status)
        torch.cuda.synchronize()
        assert int(status.item()) == 0
        results.append((out.float(), lse))
    (a, la), (b, lb) = results
    assert not torch.isnan(a).any() and not torch.isnan(la).any()
    assert ((a - b).abs() <= 2 * (2e-3 + 2.0 ** -8 * b.abs())).all()
    empty = torch.isinf(lb)
    assert torch.equal(empty, torch.isinf(la))
    assert ((la - lb).abs()[~empty] <= 4e-3).all()


def test_without_a_workspace_nothing_is_cut():
    q, kv, table, ctx = _problem(80, 128, "any", 3)
    idx = torch.arange(PAGES * 64, dtype=torch.int32, device="cuda").expand(80, -1).contiguous()
    results = []
    for splits in (0, 1):
        d = B.make_desc(80, 128, 80 * PAGES, PAGES, PAGES * 64, 0.07, num_splits=splits)
        out, lse = torch.empty((80, 128, 512), dtype=torch.bfloat16, device="cuda"), torch.empty((80, 128), device="cuda")
        B.omni_sparse_mla_decode(d, q, kv, table, idx, ctx, out, lse)
        results.append((out, lse))
    assert torch.equal(results[0][0], results[1][0]) and torch.equal(results[0][1], results[1][1])
