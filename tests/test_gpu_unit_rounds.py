"""Several work units per CTA pair (more units than pairs, none longer than 32 units of 64 tokens): every request has to come out
as it does where a pair has it alone, to the bit, since the arithmetic of a unit is the same.  Odd numbers of units, empty
selections, several rounds, the longest unit that is taken this way and the first that is not, long units one after the other on
every pair, more than a pair takes, NaNs and infinities in a unit with clean ones behind it, lengths out of range, splits, and ranges."""
import ctypes
import math

import numpy as np
import pytest
import torch

from paper_2511_22481_b200 import binding as B
from paper_2511_22481_b200 import workloads as W
from parity import check_workload, compare, oracle_subset

pytestmark = pytest.mark.gpu
SCALE = 1.0 / math.sqrt(192.0)


def _form(d):
    """2: several units per pair, 0: one."""
    return B.load().omni_internal_pair_form(ctypes.byref(d), torch.cuda.get_device_properties(0).multi_processor_count, 33)


def _workload(batch, heads, most, seed, least=0):
    rng = np.random.default_rng(seed)
    lengths = rng.integers(least * 64, most * 64 + 1, batch)
    if least == 0:
        lengths[:4] = [0, 1, 64 * most, 64 * (most - 1) + 1]
    lists = [rng.permutation(int(n)) if n % 3 == 0 else np.arange(n) for n in lengths]
    pages = [most] * batch
    return W._pack("rounds", seed, heads, pages, W._shuffled_tables(rng, pages, True),
                   [np.asarray(x, dtype=np.int32) for x in lists], "cuda", dict(kind="custom"))


def _alone(w, plan, reqs, sel_len=None):
    """The requests of a workload in calls of few, a unit to a pair: what `plan` has for them is the same, NaNs included."""
    reqs, sel_len = list(reqs), w.sel_len if sel_len is None else sel_len
    for at in range(0, len(reqs), 64):                        # (few heads: enough requests to stay on this kernel)
        some = torch.tensor(reqs[at:at + 64], device="cuda")
        n = len(some)
        d = B.make_desc(n, w.heads, w.num_pages, w.page_table.shape[1], w.sel_idx.shape[1], w.scale, num_splits=1)
        assert _form(d) != 2
        out = torch.full((n, w.heads, 512), float("nan"), dtype=torch.bfloat16, device="cuda")
        lse = torch.full((n, w.heads), float("nan"), device="cuda")
        part = [t[some].contiguous() for t in (w.q, w.page_table, w.sel_idx, sel_len)]
        B.omni_sparse_mla_decode(d, part[0], w.kv_cache, part[1], part[2], part[3], out, lse)
        torch.cuda.synchronize()
        for got, want in ((plan.out[some], out), (plan.lse[some], lse)):
            assert torch.equal(torch.isnan(got), torch.isnan(want))
            assert torch.equal(torch.nan_to_num(got, nan=0.), torch.nan_to_num(want, nan=0.))


@pytest.mark.parametrize("batch,heads,most,least", [(75, 128, 32, 0), (75, 128, 33, 0), (148, 128, 3, 0), (149, 65, 18, 0), (256, 16, 9, 0),
                                                    (160, 128, 32, 19), (150, 33, 31, 30), (256, 127, 4, 3)])
def test_as_if_alone(batch, heads, most, least):
    w = _workload(batch, heads, most, batch + most, least)
    plan = B.plan_for(w, num_splits=1)
    assert _form(plan.desc) == (2 if most <= 32 else 0)
    plan.run(w.q, w.kv_cache, w.page_table, w.sel_idx, w.sel_len)
    _alone(w, plan, range(batch))
    assert int(plan.status.item()) == 0


@pytest.mark.parametrize("batch,heads,most", [(256, 128, 2), (170, 96, 7)])
@pytest.mark.parametrize("bad", ["nan", "inf"])
def test_nothing_passes_from_unit_to_unit(batch, heads, most, bad):
    """Every third request has a NaN or an infinity among its values or its scores, every seventh a length out of range."""
    w = _workload(batch, heads, most, 5 * batch + most, 1)
    value = float(bad)
    for b in range(0, batch, 3):                              # a value column, a score column, q
        page = int(w.page_table[b, int(w.sel_idx[b, 0]) // 64])
        if b % 9 == 6:
            w.q[b, b % heads, 7] = value
        else:
            w.kv_cache[page, int(w.sel_idx[b, 0]) % 64, 300 if b % 9 else 570] = value
    lengths = w.sel_len.clone()
    lengths[3::7] = w.sel_idx.shape[1] + 1
    lengths[5::14] = -1
    plan = B.plan_for(w, num_splits=1)
    assert _form(plan.desc) == 2
    plan.run(w.q, w.kv_cache, w.page_table, w.sel_idx, lengths)
    torch.cuda.synchronize()
    assert int(plan.status.item()) == B.OMNI_DEV_BAD_INDEX
    _alone(w, plan, range(batch), lengths)
    clean = [b for b in range(batch) if b % 3 and b % 7 != 3 and b % 14 != 5][::batch // 12]
    want_out, want_lse, _ = oracle_subset(w, clean, [0, heads - 1])
    at = torch.tensor(clean)
    compare(plan.out.cpu()[at][:, [0, heads - 1]], plan.lse.cpu()[at][:, [0, heads - 1]], want_out, want_lse, "clean neighbours")


def test_two_streams_and_a_graph():
    """Launches that run beside one another, and replayed ones, deal out their own units."""
    ws = [_workload(120, 128, 10, 1), _workload(200, 64, 5, 2)]
    plans = [B.plan_for(w, num_splits=1) for w in ws]
    runs = [lambda p=p, w=w: p.run(w.q, w.kv_cache, w.page_table, w.sel_idx, w.sel_len) for p, w in zip(plans, ws)]
    want = []
    for p, run in zip(plans, runs):
        assert _form(p.desc) == 2
        run()
        torch.cuda.synchronize()
        want.append((p.out.clone(), p.lse.clone()))
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        runs[0]()
    streams = [torch.cuda.Stream() for _ in ws]
    for p in plans:
        p.out.fill_(float("nan"))
        p.lse.fill_(float("nan"))
    torch.cuda.synchronize()
    for _ in range(20):
        with torch.cuda.stream(streams[0]):
            graph.replay()
        with torch.cuda.stream(streams[1]):
            runs[1]()
    torch.cuda.synchronize()
    for p, (out, lse) in zip(plans, want):
        assert torch.equal(p.out, out) and torch.equal(p.lse, lse) and int(p.status.item()) == 0


@pytest.mark.parametrize("batch,splits", [(40, 4), (80, 2), (100, 13), (130, 20)])
def test_splits(batch, splits):
    w = _workload(batch, 40, 12, splits)
    assert _form(B.plan_for(w, num_splits=splits).desc) == 2
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
