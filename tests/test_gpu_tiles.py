"""The paired-CTA kernel at the edges of its tiles: 128 tokens in two units of 64, K refilled in three groups, three
score buffers.  Numbers of units around every multiple of those, odd ones (the second CTA then has no
K rows in the last tile), partial last units, whole pages mixed with scattered ones, and a peaked softmax that
moves the reference in late tiles."""
import numpy as np
import pytest
import torch

from paper_2511_22481_b200 import binding as B
from paper_2511_22481_b200 import workloads as W
from parity import LSE_TOL, check_workload, oracle_subset, run_gpu

pytestmark = pytest.mark.gpu
DEV = "cuda"


def _lists(name, seed, heads, lists, ctx_pages):
    rng = np.random.default_rng(seed)
    pages = [ctx_pages] * len(lists)
    return W._pack(name, seed, heads, pages, W._shuffled_tables(rng, pages, True),
                   [np.asarray(x, dtype=np.int32) for x in lists], DEV, dict(kind="custom"))


@pytest.mark.parametrize("splits", [1, 2, 3])
def test_every_small_number_of_units(splits):
    lengths = [64 * u + d for u in range(0, 19) for d in (0, 1, 63)][1:]
    lists = [np.arange(n) for n in lengths]
    w = _lists("units", 5, 96, lists, 20)
    check_workload(w, 0, num_splits=splits, what="units S=%d" % splits)


@pytest.mark.parametrize("splits", [1, 2])
@pytest.mark.parametrize("heads", [40, 128])
def test_whole_and_scattered_units_in_turn(splits, heads):
    """Every pattern of gathered and boxed units over four units, then a ragged tail."""
    rng = np.random.default_rng(11)
    lists = []
    for pattern in range(16):
        parts = []
        for u in range(9):
            page = np.arange(64) + 64 * (2 * u + 1)
            scattered = (pattern >> (u % 4)) & 1
            parts.append(rng.permutation(page) if scattered else page)
        lists.append(np.concatenate(parts + [np.arange(pattern)]))
    w = _lists("mixed", 6, heads, lists, 20)
    check_workload(w, 0, num_splits=splits, what="mixed H=%d S=%d" % (heads, splits))


@pytest.mark.parametrize("flags", [0, B.OMNI_FLAG_FUSED_MERGE, B.OMNI_FLAG_NO_CLUSTER_MERGE])
def test_reference_maximum_moves_in_late_tiles(flags):
    """Rows that grow along the context: the running maximum leaves its window again and again."""
    n = 64 * 13 + 7
    w = _lists("growing", 7, 128, [np.arange(n), np.arange(n)[::-1].copy(), np.random.default_rng(1).permutation(n)], 14)
    grow = torch.linspace(0.2, 6.0, 14 * 64, device=DEV)
    rows = (w.page_table.long()[:, :, None] * 64 + torch.arange(64, device=DEV)).view(3, -1)
    flat = w.kv_cache.view(-1, 576)
    for b in range(3):
        flat[rows[b]] = (flat[rows[b]].float() * grow[:, None]).to(torch.bfloat16)
    ref_out, ref_lse, _ = oracle_subset(w)
    # A few large tokens carry each row, so the parity tests' absolute term does not apply.  What the number
    # formats allow: bf16 has 7 explicit fraction bits, so rounding to nearest moves a value by at most
    # 2^-8 of it; rounding every weight moves out by at most 2^-8 sum_j p_j |v_j|, rounding out by 2^-8 |out|;
    # fp32 sums and the exponential add parts in 10^5.
    kv = torch.stack([flat[rows[b]][w.sel_idx[b].long()] for b in range(3)]).double()
    prob = torch.softmax(torch.einsum("bhc,bjc->bhj", w.q.double(), kv) * w.scale, dim=-1)
    spread = torch.einsum("bhj,bjd->bhd", prob, kv[:, :, :512].abs()).cpu().numpy()
    bound = 2.0 ** -8 * (spread + np.abs(ref_out)) + 1e-4 * spread
    for splits in (1, 2):
        plan = run_gpu(w, flags=flags, num_splits=splits)
        assert int(plan.status.item()) == 0
        err = np.abs(plan.out.double().cpu().numpy() - ref_out)
        assert np.all(err <= bound), (splits, float((err / bound).max()))
        assert np.all(np.abs(plan.lse.double().cpu().numpy() - ref_lse) <= LSE_TOL)
