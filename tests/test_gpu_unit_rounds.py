"""Several work units per CTA pair (more units than pairs, none longer than 32 units of 64 tokens): every request has to come out
as it does where a pair has it alone, to the bit, since the arithmetic of a unit is the same.  Odd numbers of units, empty
selections, several rounds, more units than a pair takes (then there are more pairs), the longest unit that is
taken this way and the first that is not, splits, and ranges."""
import math

import numpy as np
import pytest
import torch

from paper_2511_22481_b200 import binding as B
from paper_2511_22481_b200 import workloads as W
from parity import check_workload

pytestmark = pytest.mark.gpu
SCALE = 1.0 / math.sqrt(192.0)


def _workload(batch, heads, most, seed):
    rng = np.random.default_rng(seed)
    lengths = rng.integers(0, most * 64 + 1, batch)
    lengths[:4] = [0, 1, 64 * most, 64 * (most - 1) + 1]
    lists = [rng.permutation(int(n)) if n % 3 == 0 else np.arange(n) for n in lengths]
    pages = [most] * batch
    return W._pack("rounds", seed, heads, pages, W._shuffled_tables(rng, pages, True),
                   [np.asarray(x, dtype=np.int32) for x in lists], "cuda", dict(kind="custom"))


@pytest.mark.parametrize("batch,heads,most", [(75, 128, 32), (75, 128, 33), (148, 128, 3), (149, 65, 18), (256, 16, 9)])
def test_as_if_alone(batch, heads, most):
    w = _workload(batch, heads, most, batch + most)
    plan = B.plan_for(w, num_splits=1)
    plan.run(w.q, w.kv_cache, w.page_table, w.sel_idx, w.sel_len)
    for at in range(0, batch, 64):                            # (few heads: enough requests to stay on this kernel)
        n = min(64, batch - at)
        d = B.make_desc(n, heads, w.num_pages, w.page_table.shape[1], w.sel_idx.shape[1], w.scale, num_splits=1)
        out, lse = torch.full_like(plan.out[:n], float("nan")), torch.full_like(plan.lse[:n], float("nan"))
        part = [t[at:at + n].contiguous() for t in (w.q, w.page_table, w.sel_idx, w.sel_len)]
        B.omni_sparse_mla_decode(d, part[0], w.kv_cache, part[1], part[2], part[3], out, lse)
        torch.cuda.synchronize()
        assert torch.equal(out, plan.out[at:at + n]) and torch.equal(lse, plan.lse[at:at + n])
    assert int(plan.status.item()) == 0


@pytest.mark.parametrize("batch,splits", [(40, 4), (80, 2), (100, 13), (130, 20)])
def test_splits(batch, splits):
    w = _workload(batch, 40, 12, splits)
    check_workload(w, 0, num_splits=splits, reqs=[0, 1, 2, 3, batch // 2, batch - 1], what="B=%d S=%d" % (batch, splits))


@pytest.mark.parametrize("rolling", [False, True])
def test_ranges(rolling):
    batch, heads, sizes = 100, 72, (100, 900)
    gen = torch.Generator(device="cuda")
    gen.manual_seed(4)
    pages = B.omni_rolling_pages_per_request(*sizes) if rolling else 40
    table = torch.randperm(batch * pages, generator=gen, device="cuda").int().view(batch, pages)
    kv = torch.empty((batch * pages, 64, 576), dtype=torch.bfloat16, device="cuda").normal_(0, 0.5, generator=gen)
    q = torch.empty((batch, heads, 576), dtype=torch.bfloat16, device="cuda").normal_(0, 0.5, generator=gen)
    ctx = torch.randint(0, 40 * 64, (batch,), generator=gen, device="cuda", dtype=torch.int32)
    decode = B.omni_sparse_mla_decode_rolling if rolling else B.omni_sparse_mla_decode_sink_recent

    def run(a, b):
        d = B.make_desc(b - a, heads, batch * pages, pages, sum(sizes), SCALE, num_splits=1)
        out = torch.full((b - a, heads, 512), float("nan"), dtype=torch.bfloat16, device="cuda")
        lse = torch.full((b - a, heads), float("nan"), device="cuda")
        status = torch.zeros((1,), dtype=torch.int32, device="cuda")
        decode(d, q[a:b].contiguous(), kv, table[a:b].contiguous(), ctx[a:b].contiguous(), *sizes, out, lse, None, status)
        torch.cuda.synchronize()
        assert int(status.item()) == 0
        return out, lse

    out, lse = run(0, batch)
    for a, b in ((0, 50), (50, 100)):
        alone = run(a, b)
        assert torch.equal(out[a:b], alone[0]) and torch.equal(lse[a:b], alone[1])
