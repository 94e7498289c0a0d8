"""Batched lookups in maps of 32-byte buckets just below and from 256 MB on, where a
run's lookups read keys and values together, two such tables in one phase, against
lookups of one key per lane group."""
import pytest
import torch

from paper_1908_05936_gb300 import _lib as L
from paper_1908_05936_gb300.batch import Batch, Item
from paper_1908_05936_gb300.table import VAL_BYTES, Table

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("kind", (L.MAP_I64_I32, L.MAP_U64_U64))
@pytest.mark.parametrize("n", (1, 33, 70001))
def test_lookups_on_both_sides_of_256_mb(kind, n):
    width = torch.int64 if VAL_BYTES[kind] == 8 else torch.int32
    g = torch.Generator(device="cuda").manual_seed(n)
    tabs = [Table(kind, slots, bucket_bytes=32) for slots in ((1 << 24) - 3, (1 << 24) + 1)]
    try:
        keys = torch.randint(-(1 << 62), 1 << 62, (1 << 23,), generator=g, device="cuda")
        keys[:3] = torch.tensor([-1, -2, -3], device="cuda")
        q = torch.cat([keys[:n // 2 + 1], keys[:n // 2 + 1] + 1])[:n].contiguous()
        outs = []
        for t in tabs:
            t.insert(keys, (keys >> 20).to(width), status=False)
            t.erase(keys[5::7].contiguous(), status=False)
            outs += [(torch.empty(n, dtype=torch.uint8, device="cuda"), torch.empty(n, dtype=width, device="cuda")),
                     (torch.empty(n, dtype=torch.uint8, device="cuda"), None)]
        b = Batch([Item(t, L.OP_FIND, q, None, *o) for t, o in zip([tabs[0]] * 2 + [tabs[1]] * 2, outs)])
        b.launch()
        torch.cuda.synchronize()
        b.close()
        for t, (found, vals) in zip([tabs[0]] * 2 + [tabs[1]] * 2, outs):
            t.set_launch(L.OP_FIND, keys_per_group=1)
            f, v = t.find(q)
            assert torch.equal(found, f) and (vals is None or torch.equal(vals, v))
    finally:
        for t in tabs:
            t.close()
