"""The 8-bit kernel at the edges of its tiles (128 tokens in two units, two K stages, three V stages, rings of five
tiles): every small number of units, whole and scattered units in turn, scales that differ from row to row."""
import numpy as np
import pytest
import torch

from paper_2511_22481_b200 import workloads as W
from parity import check_workload_q8

pytestmark = pytest.mark.gpu
DEV = "cuda"


def _lists(name, seed, heads, lists, ctx_pages):
    rng = np.random.default_rng(seed)
    pages = [ctx_pages] * len(lists)
    w = W._pack(name, seed, heads, pages, W._shuffled_tables(rng, pages, True),
                [np.asarray(x, dtype=np.int32) for x in lists], DEV, dict(kind="custom"))
    gen = torch.Generator(device=DEV).manual_seed(seed)
    # a scale of its own for every row: powers of two, exact in bf16
    factor = torch.exp2(torch.randint(-2, 2, w.kv_cache.shape[:2], generator=gen, device=DEV).float())
    w.kv_cache.mul_(factor[..., None].to(torch.bfloat16))
    return w


@pytest.mark.parametrize("splits", [1, 2, 3])
def test_every_small_number_of_units(splits):
    lengths = [64 * u + d for u in range(0, 19) for d in (0, 1, 63)][1:]
    w = _lists("q8 units", 5, 96, [np.arange(n) for n in lengths], 20)
    check_workload_q8(w, 0, num_splits=splits, what="q8 units S=%d" % splits)


@pytest.mark.parametrize("splits", [1, 2])
def test_whole_and_scattered_units_in_turn(splits):
    rng = np.random.default_rng(11)
    lists = []
    for pattern in range(16):
        parts = []
        for u in range(9):
            page = np.arange(64) + 64 * (2 * u + 1)
            parts.append(rng.permutation(page) if (pattern >> (u % 4)) & 1 else page)
        lists.append(np.concatenate(parts + [np.arange(pattern)]))
    w = _lists("q8 mixed", 6, 128, lists, 20)
    check_workload_q8(w, 0, num_splits=splits, what="q8 mixed S=%d" % splits)
