"""The split plan where it weighs a merge in a cluster, the merge kernel and the number of partial results
against each other (148 SMs, 33 resident merging clusters).  The counts are the fastest, or within 4 % of
it, of all those measured at the shape."""
import ctypes
import math

import pytest
import torch

from paper_2511_22481_b200 import binding as B
from paper_2511_22481_b200 import build as builder


@pytest.mark.parametrize("batch,heads,units,want", [
    (4, 128, 8, (1, 1)),        # the longest request that is never cut
    (4, 128, 9, (2, 1)),        # the shortest that is
    (16, 128, 16, (2, 1)), (24, 128, 33, (2, 1)),
    (33, 128, 33, (2, 1)),      # the last batch whose clusters are all resident
    (34, 128, 12, (1, 1)),      # the first whose are not
    (4, 128, 16, (8, 2)),       # few partial results
    (36, 128, 64, (2, 2)),      # partial results pay all the same
    (48, 128, 64, (1, 1)),
    (4, 16, 4, (4, 2)),         # single-CTA kernel
])
def test_split_choice(batch, heads, units, want):
    builder.build()
    d = B.make_desc(batch, heads, batch * units, units, units * 64, 1.0 / math.sqrt(192.0))
    assert B.omni_sparse_mla_plan_query(d, 148, 33) == want


@pytest.mark.parametrize("batch,heads,units,splits,flags,want", [
    (75, 128, 32, 1, 0, 2), (75, 128, 33, 1, 0, 0), (74, 128, 32, 1, 0, 0),       # more units than pairs, none longer than 32
    (256, 128, 18, 1, 0, 2), (257, 128, 18, 1, 0, 0),                             # as many as the kernel ranks
    (40, 128, 64, 2, 0, 2), (33, 128, 64, 2, 0, 1), (100, 40, 12, 13, 0, 2),      # splits; a merge in a cluster
    (100, 128, 12, 3, B.OMNI_FLAG_FUSED_MERGE, 0),                                # a merge by the last CTA
    (76, 128, 64, 0, 0, 0),                                                       # only the last two requests are cut
    (4, 16, 4, 0, 0, -1),                                                         # single-CTA kernel
])
def test_units_per_pair(batch, heads, units, splits, flags, want):
    builder.build()
    d = B.make_desc(batch, heads, batch * units, units, units * 64, 1.0 / math.sqrt(192.0), num_splits=splits, flags=flags)
    assert B.load().omni_internal_pair_form(ctypes.byref(d), 148, 33) == want


@pytest.mark.gpu
@pytest.mark.parametrize("batch,heads,units", [(4, 128, 9), (3, 128, 11), (4, 16, 4)])
def test_short_selections_need_no_workspace(batch, heads, units):
    """Without a workspace the requests stay whole: the bits of one forced split."""
    from paper_2511_22481_b200 import workloads as W
    w = W.token_topk("short", 5, batch, heads, 32, units * 64, "cuda")
    ref = B.plan_for(w, num_splits=1)
    ref.run(w.q, w.kv_cache, w.page_table, w.sel_idx, w.sel_len)
    d = B.plan_for(w)
    assert d.splits > 1
    out, lse = torch.full_like(ref.out, float("nan")), torch.full_like(ref.lse, float("nan"))
    B.omni_sparse_mla_decode(d.desc, w.q, w.kv_cache, w.page_table, w.sel_idx, w.sel_len, out, lse)
    torch.cuda.synchronize()
    assert torch.equal(out, ref.out) and torch.equal(lse, ref.lse)
