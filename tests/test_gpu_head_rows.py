"""The paired-CTA kernel with every kind of uneven head count: the two CTAs of a pair share the heads evenly, so either has
ceil(heads / 2) rows, of which the second may lack one, q comes in boxes of that many rows, and the other rows are zeros
that nobody stores.  Forty requests, so that few heads are on this kernel too; two splits merge in a cluster, three in
the merge kernel."""
import numpy as np
import pytest

from paper_2511_22481_b200 import binding as B
from paper_2511_22481_b200 import workloads as W
from parity import check_workload

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("splits,batch", [(1, 40), (2, 30), (3, 40)])
@pytest.mark.parametrize("heads", [1, 2, 9, 33, 64, 65, 95, 127])
def test_uneven_heads(heads, splits, batch):
    rng = np.random.default_rng(heads)
    lists = [rng.permutation(11 * 64)[:n] if n % 2 else np.arange(n) for n in rng.integers(1, 11 * 64, batch)]
    lists[0] = np.arange(11 * 64)
    pages = [11] * batch
    w = W._pack("head rows", 12, heads, pages, W._shuffled_tables(rng, pages, True),
                [np.asarray(x, dtype=np.int32) for x in lists], "cuda", dict(kind="custom"))
    check_workload(w, 0, num_splits=splits, what="H=%d S=%d" % (heads, splits))
    check_workload(w, B.OMNI_FLAG_FUSED_MERGE, num_splits=splits, what="fused H=%d S=%d" % (heads, splits))
