"""The host-buffer entry point in each of its forms: pinned buffers used in place (one, two and four
parts, index arrays at once or by part) and copies for any other host memory.  Every form gives the bits of
the device entry point run on the same parts' sizes, up to the split plan, so the oracle decides."""
import pytest
import torch

from paper_2511_22481_b200 import binding as B
from paper_2511_22481_b200 import workloads as W
from parity import compare, oracle_subset

pytestmark = pytest.mark.gpu
DEV = "cuda"


def _host(t, kind, offset=2):
    if kind == "pinned":
        return t.cpu().pin_memory()
    if kind == "pageable":
        return t.cpu()
    flat = torch.empty(t.numel() + offset, dtype=t.dtype).pin_memory()     # pinned, but not at a 16-byte boundary
    flat[offset:].copy_(t.cpu().reshape(-1))
    return flat[offset:].view(t.shape)


def _run(w, kinds, reqs=None):
    desc = B.make_desc(w.batch, w.heads, w.num_pages, w.max_pages_per_req, w.max_sel, w.scale)
    staging = torch.empty(B.omni_sparse_mla_host_staging_bytes(desc), dtype=torch.uint8, device=DEV)
    ws = torch.empty(max(1, B.omni_sparse_mla_workspace_bytes(desc)), dtype=torch.uint8, device=DEV)
    ins = [_host(t, k) for t, k in zip((w.q, w.page_table, w.sel_idx, w.sel_len), kinds)]
    out = _host(torch.full((w.batch, w.heads, 512), float("nan"), dtype=torch.bfloat16), kinds[4])
    lse = _host(torch.full((w.batch, w.heads), float("nan")), kinds[5])
    status = torch.zeros(1, dtype=torch.int32, device=DEV)
    for _ in range(2):                                   # back-to-back calls reuse the staging buffer
        B.omni_sparse_mla_decode_host(desc, ins[0], w.kv_cache, *ins[1:], out, lse, staging, ws, status)
    torch.cuda.current_stream().synchronize()
    assert int(status.item()) == 0
    ref_out, ref_lse, _ = oracle_subset(w, reqs=reqs)
    pick = slice(None) if reqs is None else reqs
    compare(out[pick], lse[pick], ref_out, ref_lse, "host %s" % (kinds,))


@pytest.mark.parametrize("batch,heads", [(1, 16), (2, 128), (3, 128), (4, 128), (7, 128), (8, 128), (9, 65), (12, 128), (13, 128), (15, 128), (33, 65)])
def test_pinned_parts(batch, heads):
    _run(W.token_topk("host", 11 + batch, batch, heads, 8, 301, DEV), ["pinned"] * 6)


@pytest.mark.parametrize("batch", [3, 14])
@pytest.mark.parametrize("odd", range(6))
def test_one_buffer_that_cannot_be_used_in_place(batch, odd):
    for kind in ("pageable", "shifted"):
        kinds = ["pinned"] * 6
        kinds[odd] = kind
        _run(W.token_topk("host", 5, batch, 128, 6, 200, DEV), kinds, reqs=[0, batch // 2, batch - 1])


def test_large_index_arrays_come_by_part():
    """Sixteen requests of 20000 positions: 1.3 MB of indices, and kernels that outlast the transfers."""
    _run(W.dense("host dense", 3, 16, 128, 313, DEV), ["pinned"] * 6, reqs=[0, 7, 8, 15])


def test_large_index_arrays_in_four_parts():
    w = W.token_topk("host wide", 4, 24, 128, 512, 300, DEV)
    wide = torch.full((24, 20000), -1, dtype=torch.int32, device=DEV)
    wide[:, :300] = w.sel_idx
    w.sel_idx, w.max_sel = wide, 20000
    _run(w, ["pinned"] * 6, reqs=[0, 9, 10, 23])
