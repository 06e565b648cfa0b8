"""The single-CTA kernel at the edges of its tiles and of its head rows: partial rows leave eight rows at a time, each
warp owns sixteen, scores start on the first third of a tile's panels, and a split may be empty."""
import numpy as np
import pytest

from paper_2511_22481_b200 import workloads as W
from parity import check_workload

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("heads", [1, 8, 9, 16, 17, 31, 32])
@pytest.mark.parametrize("splits", [1, 2, 5, 13])
def test_head_rows_and_tiles(heads, splits):
    rng = np.random.default_rng(heads)
    lengths = [1, 63, 64, 65, 190, 64 * 13, 64 * 13 + 1]          # with 5 and 13 splits some are empty
    lists = [np.arange(n) for n in lengths] + [rng.permutation(16 * 64)[:300]]
    pages = [16] * len(lists)
    w = W._pack("few heads", 9, heads, pages, W._shuffled_tables(rng, pages, True),
                [np.asarray(x, dtype=np.int32) for x in lists], "cuda", dict(kind="custom"))
    check_workload(w, 0, num_splits=splits, what="H=%d S=%d" % (heads, splits))


@pytest.mark.parametrize("batch,tiles", [(1, 40), (1, 41), (2, 80), (2, 81), (1, 192)])
def test_either_side_of_forty_tiles_a_request(batch, tiles):
    """The longest selection that few requests of few heads take to this kernel (40 tiles for each of them), and the first that
    pairs serve."""
    rng = np.random.default_rng(tiles)
    lists = [rng.permutation(tiles * 64), np.arange(tiles * 64 - 63)][:batch]
    pages = [tiles] * batch
    w = W._pack("forty", 10, 16, pages, W._shuffled_tables(rng, pages, True),
                [np.asarray(x, dtype=np.int32) for x in lists], "cuda", dict(kind="custom"))
    check_workload(w, 0, what="B=%d tiles=%d" % (batch, tiles))
