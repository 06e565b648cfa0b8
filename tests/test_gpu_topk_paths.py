"""The selection producer's two ways to a threshold (a bound from group maxima, or digit by digit over all keys)
and the edges between them, bit for bit against the oracle."""
import numpy as np
import pytest
import torch

from oracle.topk import topk_batch
from paper_2511_22481_b200 import binding as B

pytestmark = pytest.mark.gpu


def _check(scores, ctx_len, k, offset=0):
    flat = torch.zeros(scores.size + offset, device="cuda")
    s = flat[offset:].view(scores.shape)                   # a row start that is not 16-byte aligned if offset % 4
    s.copy_(torch.from_numpy(scores))
    ctx = torch.tensor(list(ctx_len), dtype=torch.int32, device="cuda")
    idx = torch.full((scores.shape[0], k), -7, dtype=torch.int32, device="cuda")
    length = torch.full((scores.shape[0],), -7, dtype=torch.int32, device="cuda")
    B.omni_topk_select(s, ctx, k, idx, length)
    want_idx, want_len = topk_batch(scores, ctx_len, k)
    assert length.cpu().numpy().tolist() == want_len.tolist()
    got = idx.cpu().numpy()
    for b, n in enumerate(want_len):
        assert np.array_equal(got[b, :n], want_idx[b, :n]), b
        assert np.all(got[b, n:] == -7)


@pytest.mark.parametrize("stride", [1023, 4096, 4099, 32768, 65541, 131072])
@pytest.mark.parametrize("share", [64, 9, 8, 7, 2, 1])
def test_more_and_fewer_groups_than_the_bound_needs(stride, share):
    """Vectors of four scores bound the search from k = stride / 8 down; above, all keys are searched."""
    rng = np.random.default_rng(stride + share)
    scores = rng.standard_normal((3, stride)).astype(np.float32)
    _check(scores, [stride, stride - 1, stride // 2], max(1, stride // share))


@pytest.mark.parametrize("offset", [0, 1, 2, 3])
def test_rows_at_any_alignment(offset):
    rng = np.random.default_rng(offset)
    for stride in (130, 4097, 30002):
        scores = rng.standard_normal((3, stride)).astype(np.float32)
        _check(scores, [stride, stride - 2, 5], 40, offset)


def test_crowded_scores():
    """More keys from the bound on than the lists hold: equal scores, few values, values one ulp apart,
    everything NaN but a few, and maxima that all sit in one bin of their leading bits."""
    rng = np.random.default_rng(5)
    n, k = 50000, 700
    rows = [np.full(n, 1.5), rng.integers(0, 3, n) * 1.0,
            (np.float32(1).view(np.uint32) + rng.integers(0, 6000, n).astype(np.uint32)).view(np.float32),
            np.where(rng.random(n) < 0.01, rng.standard_normal(n), np.nan),
            rng.uniform(1.0, 1.2, n), -np.abs(rng.standard_normal(n)) * 1e-40, np.where(rng.random(n) < 0.5, np.inf, -np.inf),
            np.concatenate([np.zeros(n - 3), [7, 8, 9]])]
    scores = np.stack([r.astype(np.float32) for r in rows])
    _check(scores, [n] * len(rows), k)
    _check(scores, [n - 17] * len(rows), 1)
    _check(scores, [n] * len(rows), n - 1)


def test_scores_in_order():
    """All the largest scores in one CTA's share, at its front or its end."""
    n = 131072
    up = np.arange(n, dtype=np.float32)
    _check(np.stack([up, up[::-1].copy()]), [n, n], 2048)
