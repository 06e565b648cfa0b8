"""Both sides of the rules that pick a kernel: single CTA or pair by heads and size, one or four thread
groups in the merge.  Everything is compared with the oracle under the parity tolerances."""
import numpy as np
import pytest
import torch

import oracle
from paper_2511_22481_b200 import binding as B
from paper_2511_22481_b200 import workloads as W
from parity import check_workload

pytestmark = pytest.mark.gpu
DEV = "cuda"


@pytest.mark.parametrize("heads", [1, 32, 33, 63, 64])
@pytest.mark.parametrize("batch,tokens", [(1, 64), (3, 500), (74, 129), (75, 129)])
def test_few_heads_on_both_sides_of_the_rule(heads, batch, tokens):
    """74 requests of three tiles are 148 two-tile units, 75 are 150; 33 heads never run on a single CTA."""
    w = W.token_topk("few heads", 7 + heads, batch, heads, 9, tokens, DEV)
    reqs = sorted({0, batch // 2, batch - 1})
    for splits in (0, 2):
        check_workload(w, 0, num_splits=splits, reqs=reqs, what="H=%d B=%d N=%d S=%d" % (heads, batch, tokens, splits))


@pytest.mark.parametrize("heads", [5, 64])
def test_few_heads_fused_merge(heads):
    w = W.token_topk("few heads fused", 3, 80, heads, 10, 600, DEV)
    check_workload(w, B.OMNI_FLAG_FUSED_MERGE, num_splits=3, reqs=[0, 41, 79], what="fused H=%d" % heads)


@pytest.mark.parametrize("splits", [1, 4, 5, 31, 32, 33, 70])
@pytest.mark.parametrize("batch,heads", [(1, 3), (6, 74), (6, 75)])
def test_merge_of_any_number_of_splits(splits, batch, heads):
    """(6, 74): as many blocks as three per SM, (6, 75): more.  Empty splits carry rows of NaN, which must
    not be read; fp32 sums of at most 70 terms, results rounded to bf16 (half an ulp: at most 2^-8 of the value)."""
    rng = np.random.default_rng(splits)
    part = rng.standard_normal((batch, splits, heads, 512)).astype(np.float32)
    lse = (rng.standard_normal((batch, splits, heads)) * 3).astype(np.float32)
    empty = rng.random((batch, splits, heads)) < 0.2
    empty[0, :, 0] = True
    lse[empty] = -np.inf
    part[empty] = np.nan
    counts = np.full((batch,), splits, dtype=np.int32)
    counts[-1] = max(0, splits - 1)
    want, want_lse = oracle.splitkv_combine(np.where(empty[..., None], 0.0, part).astype(np.float64), lse.astype(np.float64), counts)
    desc = B.make_desc(batch, heads, 4, 4, 64, 0.1)
    out = torch.full((batch, heads, 512), float("nan"), dtype=torch.bfloat16, device=DEV)
    out_lse = torch.full((batch, heads), float("nan"), device=DEV)
    B.omni_sparse_mla_combine(desc, splits, torch.from_numpy(part).to(DEV), torch.from_numpy(lse).to(DEV),
                              torch.from_numpy(counts).to(DEV), out, out_lse)
    got, got_lse = out.float().cpu().numpy(), out_lse.cpu().numpy()
    assert np.all(np.abs(got - want) <= 2.0 ** -8 * np.abs(want) + 1e-5)
    finite = np.isfinite(want_lse)
    assert np.array_equal(finite, np.isfinite(got_lse)) and np.all(got_lse[~finite] == -np.inf)
    assert np.all(np.abs(got_lse[finite] - want_lse[finite]) <= 1e-5)
