"""Batches whose warps take their chunks from counters (lock-step phases, runs with
blocks_per_sm) or have one each, launched twice from one graph and once through
hc_batch_run, against range calls on tables of the same contents."""
import ctypes

import pytest
import torch

from paper_1908_05936_gb300 import _lib as L
from paper_1908_05936_gb300.batch import Batch, Item
from paper_1908_05936_gb300.table import Table
from test_gpu_bulk import keys_of, vals_of
from test_zz_no_alloc import _item_array

pytestmark = pytest.mark.gpu

SLOTS = (40, 5000, 128, 70001, 300)


def items_for(kind):
    tabs, items = [], []
    for x, slots in enumerate(SLOTS):
        t = Table(kind, slots, bucket_bytes=64)
        k = keys_of(torch.arange(x << 20, (x << 20) + slots // 2 + 1, device="cuda"), kind)
        q = torch.cat([k, k + 1])
        out = [torch.empty(a.numel(), dtype=torch.uint8, device="cuda") for a in (k, q, k[::3])]
        w = torch.empty_like(q) if kind == L.MAP_U64_U64 else None
        tabs.append(t)
        items += [Item(t, L.OP_INSERT, k, vals_of(k, kind), out[0]), Item(t, L.OP_FIND, q, None, out[1], w),
                  Item(t, L.OP_ERASE, k[::3].contiguous(), None, out[2])]
    return tabs, items


@pytest.mark.parametrize("kind", (L.SET_U64, L.MAP_U64_U64))
@pytest.mark.parametrize("kpt", (1, 2, 4, 8))
@pytest.mark.parametrize("per_sm", (0, 1, 3))
@pytest.mark.parametrize("how", ("graph", "run"))
def test_grids(kind, kpt, per_sm, how):
    tabs, items = items_for(kind)
    ref_tabs, ref = items_for(kind)
    try:
        if how == "graph":
            b = Batch(items, keys_per_group=kpt, blocks_per_sm=per_sm, use_graph=True)
        else:
            lib = tabs[0].lib
            scratch = torch.empty(int(lib.hc_batch_scratch_bytes(len(items))) + 256, dtype=torch.uint8, device="cuda")
            cfg = L.BatchConfig(0, kpt, 0, per_sm, 0, 0)
        for _ in range(2):
            if how == "graph":
                b.launch()
            else:
                base = (scratch.data_ptr() + 255) // 256 * 256
                L.check(lib.hc_batch_run(_item_array(items), len(items), ctypes.byref(cfg), base,
                                         scratch.numel() - (base - scratch.data_ptr()),
                                         torch.cuda.current_stream().cuda_stream))
            torch.cuda.synchronize()
            for x, it in enumerate(ref):
                if it.op == L.OP_INSERT:
                    want = it.table.insert(it.keys, it.vals)
                    assert torch.equal(items[x].out, want)
            for x, it in enumerate(ref):
                if it.op == L.OP_FIND:
                    f, w = it.table.find(it.keys)
                    assert torch.equal(items[x].out, f) and (w is None or torch.equal(items[x].vals_out, w))
            for x, it in enumerate(ref):
                if it.op == L.OP_ERASE:
                    assert torch.equal(items[x].out, it.table.erase(it.keys))
        for t, r in zip(tabs, ref_tabs):
            assert t.size() == r.size() and t.status() == L.OK
        if how == "graph":
            b.close()
    finally:
        for t in tabs + ref_tabs:
            t.close()
